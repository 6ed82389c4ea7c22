// kernels.h -- host-side launchers of the libsoma kernels (internal).
#pragma once

#include <string>
#include <vector>

#include "common.cuh"

namespace soma {

// Launches a kernel of the cycle (one that begins with chained_begin) so that it
// is set up while the kernel before it in the stream still runs: a cycle is two
// or three kernels, and the gap between two of them is a microsecond of idle
// SMs.  For kernels of one block per SM and the field kernels: a kernel of several
// blocks per SM finds them spread unevenly, or the SM's shared memory still split for
// the kernel before it (a batch of 64 systems went from 28.1 to 29.6 ms, the
// molecule-parallel iteration of 134M particles from 1.9 to 3.3 ms).
inline cudaError_t launch_chained(const void* fn, dim3 grid, dim3 block, void** args, size_t smem,
                                  cudaStream_t st) {
  cudaLaunchAttribute a;
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &a;
  c.numAttrs = 1;
  return cudaLaunchKernelExC(&c, fn, args);
}

// Launch shape of the sweep kernel for chains of N particles: Q pairs of
// particles per lane, G whole chains per 32-lane tile.
struct SweepShape {
  int Q;
  uint32_t G;
  uint64_t n_tiles;
  bool pair;  // even N <= 64: one even and one odd particle per lane
  bool strip;       // the strip layout (strip.cuh), else tiles of whole chains
  bool wide;        // every axis has two or more cells
  uint32_t units;   // strips: units per chain, chains per work item, items
  uint32_t chains;
  uint64_t n_items;
  bool big;   // 64-bit particle indices (M >= 2^32)
  int move;   // 0 uniform, 1 smart Monte Carlo, 2 learned
  bool learned_tc;  // learned move with the network on the tensor cores
  bool learned_umma;  // ... through tcgen05 (else warp-level mma.sync)
  bool molecule;      // molecule-parallel iteration
  bool chained;       // launched with launch_chained
  int block;
  int grid;
};

SweepShape sweep_shape(const Geom& g, int sm_count, int grid_dtype, int move,
                       bool learned_fp32 = false, bool learned_umma = false,
                       bool molecule = false);
cudaError_t launch_sweep_uniform(const SweepArgs& a, const SweepShape& s, int grid_dtype,
                                 int sm_count, cudaStream_t st);

// Many cycles of a small system in one cooperative launch (resident.cu).
// grid 0: the system takes the two-kernel cycle.
struct ResidentShape {
  int grid, block;
  size_t cluster_smem;   // shared memory of the one-cluster kernel (0: the cooperative one)
  uint32_t min_cycles;   // shorter calls take the two kernels
};
struct ResidentArgs {
  SweepArgs s;
  FieldArgs f;
  uint32_t* n2;        // third count buffer, cleared between launches
  unsigned* bar;       // grid barrier counter, 0 between launches
  unsigned* arrive;    // blocks that have ended, 0 between launches
  uint32_t cycles;
};
// Largest system of the resident sweep, in tiles of 64 slots per SM: two rounds of
// 32 warps.  Resident against two kernels a cycle in long calls: 27 tiles per SM 7.4
// and 9.3 us, 40 9.1 and 11.1, 61 11.0 and 11.9, 91 14.1 and 14.5 (16 cycles 234 and
// 229), 121 16.8 and 16.6.  That is for a system alone: its blocks hold their SMs for all
// cycles, and several systems on their own streams, which two kernels a cycle let in
// turn, wait for one another (four of 32,768 particles 237 us for 32 cycles, with two
// kernels 305; of 131,072 435 and 406; of 300,000 998 and 678).
constexpr uint64_t RESIDENT_TILES_PER_SM = 64;
// Fewest cycles of a call that take it: two, and one more per 16 tiles per SM.  Its
// launch and last field update cost what some cycles gain; calls back to back,
// resident against two kernels: one cycle at 3 tiles per SM 9.9 and 7.2 us, 40 16.3
// and 11.5; two at 8 14.6 and 14.8, 27 22.8 and 19.0; four at 40 42.6 and 45.3, 61 49.3
// and 47.4; eight at 61 90.6 and 95.0.
constexpr uint64_t RESIDENT_TILES_PER_CYCLE = 16;
// One cluster: 16 blocks of up to 16 warps, a tile each, and the counts three times
// in a block's shared memory (96 KB at the limit).  With 32 warps on its 16 SMs
// their issue slots are the time: 32,768 particles 4.4 us a cycle against 4.2 over
// all SMs; 13,664 2.9 against 3.9.
constexpr int CLUSTER_BLOCKS = 16;
constexpr int CLUSTER_WARPS = 16;
constexpr uint32_t CLUSTER_CELLS = 8192;
ResidentShape resident_shape(const SweepShape& s, uint32_t cells, int grid_dtype, int sm_count);
cudaError_t launch_resident(const ResidentArgs& a, const ResidentShape& s, int grid_dtype,
                            cudaStream_t st);

cudaError_t launch_init(const Geom& g, float* x, float* y, float* z, double sigma, int sm_count,
                        cudaStream_t st);
// Re-label whole chains in Morton order of the 8^3-cell block of their first
// particle: src and dst are 3-plane position buffers, keys holds n_pad >=
// n_chains (a power of two) 64-bit words of scratch.
cudaError_t launch_sort_chains(const Geom& g, const float* src, uint64_t src_plane, float* dst,
                               uint64_t dst_plane, uint64_t* keys, uint64_t n_pad, int sm_count,
                               cudaStream_t st);
// seq/arch: the per-chain type sequences of a mixture (NULL: diblocks of N_A A particles);
// alen: particles of each architecture (NULL: all N), absent slots not counted
cudaError_t launch_histogram(const Geom& g, const float* x, const float* y, const float* z,
                             uint32_t* n, int sm_count, cudaStream_t st,
                             const uint64_t* seq = nullptr, const uint8_t* arch = nullptr,
                             const uint8_t* alen = nullptr);
// the same for positions on this device, copied on the way: dst + d plane = src + d n, d < 3
cudaError_t launch_copy_check(const float* src, float* dst, uint64_t n, uint64_t plane, float lim,
                              unsigned* flag, int sm_count, cudaStream_t st);
cudaError_t launch_range_check(const float* p, uint64_t n, float lim, unsigned* flag, int sm_count,
                               cudaStream_t st);
cudaError_t launch_fields(const FieldArgs& a, unsigned* arrive, int grid_dtype, int sm_count,
                          cudaStream_t st);
cudaError_t launch_convert_fields(const void* w, int grid_dtype, float* dst, uint64_t n,
                                  cudaStream_t st);

// FP64 observables: partial sums per block into part, then one block folds
// them in a fixed order into out (device).
//   out[0] = sum over bonds |b|^2, out[1] = sum over chains |R_e|^2,
//   out[2] = sum over cells of K(c) (Eq. discrete-ham, without rho dL^3/N),
//   out[3] = max over cells of n_A + n_B.
constexpr int OBS_BLOCKS = 1024;
// part: 5 * OBS_BLOCKS doubles; out: b2, Re2 sums, K sum, max cell, external energy
cudaError_t launch_observables(const Geom& g, const float* x, const float* y, const float* z,
                               const uint32_t* n, double inv_rho, double kappaN, double chiN,
                               int hamiltonian, const float* ext, double* part, double* out,
                               cudaStream_t st);

// S(q) for k <= SQ_MAX wave vectors m (host, k x 3); tw (device) holds the FP64
// twiddles e^{-2 pi i r/n} (cos, -sin), r < n, of the three axes in turn
// (nx + ny + nz pairs); part: SQ_BLOCKS * 2 * SQ_MAX doubles of scratch.
constexpr int SQ_MAX = 32;
constexpr int SQ_BLOCKS = 512;
cudaError_t launch_structure_factor(const Geom& g, const uint32_t* n, const double* tw,
                                    const int32_t* m, int k, double* part, double* out,
                                    cudaStream_t st);

cudaError_t launch_philox(const uint32_t* ctr, const uint32_t* key, uint32_t* out, size_t n,
                          cudaStream_t st);
// out[4i..4i+3] = the three normals and ln u a smart Monte Carlo move takes
// from draw words[4i..4i+3]
cudaError_t launch_smc_draws(const uint32_t* words, float* out, size_t n, int sm_count,
                             cudaStream_t st);

cudaError_t launch_sweep_batch(const BatchArgs& a, int grid, int block, int grid_dtype,
                               cudaStream_t st);
cudaError_t launch_fields_batch(const BatchArgs& a, uint32_t total_cells, unsigned* arrive,
                                unsigned* err, int grid_dtype, int sm_count, cudaStream_t st);
int batch_kernel_blocks_per_sm(int block, int grid_dtype);

cudaError_t launch_sweep_learned(const SweepArgs& a, const SweepShape& s, int grid_dtype,
                                 const void* wq, cudaStream_t st);
cudaError_t launch_esjd_grad(const TrainArgs& t, int grid_dtype, int sm_count, cudaStream_t st);
// out[0] = sum of J, out[1] = sum of min(1, exp(log_alpha)) (FP64); part: 2 OBS_BLOCKS doubles
cudaError_t launch_train_sums(const float* J, const float* log_alpha, uint32_t n, int sm_count,
                              double* part, double* out, cudaStream_t st);
cudaError_t launch_adam(float* w, float* m, float* v, const float* grad, void* wq, float lr,
                        float b1, float b2, float eps, int step, float inv_n, cudaStream_t st);
cudaError_t launch_quantize(const float* w, void* wq, cudaStream_t st);
const void* learned_kernel_ptr(int Q, int grid_dtype);
const void* learned_tc_kernel_ptr(bool umma);
// one warp waits (at most limit polls) for an mbarrier phase nobody completes
cudaError_t launch_wait_probe(uint32_t limit, unsigned* err, cudaStream_t st);
// molecule-parallel sweep kernel for n_chains chains of N particles and its dynamic
// shared memory; molecule_grid gives its blocks and allows it that memory (call
// it before the first launch, outside stream capture)
constexpr int MOL_BLOCK = 128;
const void* molecule_kernel(uint64_t n_chains, uint32_t N, int grid_dtype, int sm_count, size_t* smem);
int molecule_grid(uint64_t n_chains, uint32_t N, int grid_dtype, int sm_count);
// smart Monte Carlo sweep kernel: pair tiles or strips (big: 64-bit indices)
const void* smc_kernel_ptr(bool strip, bool big);

// Molecules of any architecture (topology.cu): the architecture array of
// Sec. 3.2.1 and the independent sets derived from it.
// The bond lists of the array are re-encoded per particle: one 32-bit word
// with its degree, its first three partners, type, set and the number of sets,
// and a 64-bit mask of all its partners (bit j: bonded to particle j of the
// molecule) read only for particles with more than three.
struct TopoArgs {
  SweepArgs s;               // geometry, positions, fields, tile shape (G = 64/N)
  const uint64_t* pmask;     // partners of particle i of architecture a: [a*64 + i]
  const uint32_t* ptab;      // [a*64 + i]: degree, first three partners, type, set, sets
  const uint8_t* mol_arch;   // architecture of every molecule
  const uint8_t* alen;       // particles of each architecture (the slots past it are absent)
  // n_t types: type of particle i of architecture a ([a*64 + i]), the field
  // planes (n_types * cells) and the count planes of both parities
  const uint8_t* ttab;
  const float* wt;
  uint32_t* nt0;
  uint32_t* nt1;
  // architectures of at most two sets: [a*32 + rank] = table words of the
  // rank-th particles of set 0 and set 1, and particle0 | particle1 << 8 |
  // type0 << 16 | type1 << 24 (0xFF: none); lanes and molecules per warp tile
  const uint4* pair_tab;
  uint32_t pair_R, pair_G;
};
struct TopologyTables {
  std::vector<uint64_t> pmask;   // n_arch * 64
  std::vector<uint32_t> ptab;    // n_arch * 64
  std::vector<uint8_t> ttab;     // n_arch * 64, type of each particle
  uint32_t max_type = 0;
  std::vector<uint8_t> nsets;    // n_arch
  std::vector<uint64_t> seq;     // type bits (bit i: particle i is B)
  std::vector<uint32_t> bonds;   // bonds per architecture
  std::vector<uint8_t> len;      // particles per architecture (<= N; the rest absent)
};
// Checks an architecture array against a system of N particle slots per
// molecule (an architecture holds 1..N particles, the first slots of its
// molecules) and derives the tables -- an absent slot has table word 0 (no
// sets), no partners and type byte 0xFF; returns an empty string or what is
// wrong.
std::string topology_tables(const uint32_t* words, uint64_t n_words, const uint32_t* start,
                            uint32_t n_arch, uint32_t N, TopologyTables* out,
                            uint32_t n_types = 2);
// Pairs of one particle of set 0 and one of set 1 per lane; R = 0 where some
// architecture has more than two sets or a warp would hold fewer molecules than
// a tile of the general kernel.
struct TopologyPairs {
  std::vector<uint4> tab;
  uint32_t R = 0, G = 0;
};
TopologyPairs topology_pairs(const TopologyTables& T, uint32_t n_arch, uint32_t N);
int topology_pair_grid(uint64_t n_mol, uint32_t G, int sm_count);
cudaError_t launch_sweep_topology_pair(const TopoArgs& a, int grid, int grid_dtype, cudaStream_t st,
                                       bool types, bool smc);
// smc: the smart Monte Carlo move (the table s.smc_tab holds one plane per type)
int topology_grid(int grid_dtype, bool big, int sm_count, uint64_t n_tiles, bool types = false,
                  bool smc = false);
cudaError_t launch_sweep_topology(const TopoArgs& a, int grid, int grid_dtype, bool big,
                                  cudaStream_t st, bool types = false, bool smc = false);
// the molecule-parallel iteration for molecules of any architecture (N <= 64);
// the grid helper also allows the kernel its shared memory (call it before
// the first launch, outside stream capture)
int molecule_topology_grid(uint32_t N, int grid_dtype, int sm_count, uint64_t n_chains, bool types);
cudaError_t launch_molecule_topology(const TopoArgs& a, int grid, int grid_dtype, int sm_count,
                                     cudaStream_t st, bool types);
// out[0] = sum over the bonds of the architectures of |b|^2, out[1] = sum over
// the molecules of |r_last - r_0|^2 with r_last the last particle of each
// molecule's architecture (lengths alen) (FP64); part: 2 OBS_BLOCKS doubles
cudaError_t launch_topology_bonds(const Geom& g, const float* x, const float* y, const float* z,
                                  const uint64_t* pmask, const uint8_t* mol_arch,
                                  const uint8_t* alen, double* part, double* out, cudaStream_t st);

// n_t particle types (types.cu).
constexpr int TYPES_MAX = 8;
struct TypesArgs {
  Geom g;
  uint32_t* n0;              // count planes, n_types * cells each; the sweep of step s
  uint32_t* n1;              // counts into planes (s+1)&1
  float* w;                  // field planes, n_types * cells
  float4* tab;               // table of a smart Monte Carlo sweep, n_types * cells (or NULL)
  unsigned long long* d_sweep;
  uint32_t n_types;
  int after_sweep;           // as FieldArgs
  int hamiltonian;           // 0: K^0_inter, 1: K^1_inter
  float inv_rho;             // 1/(rho_0 dL^3)
  float kappa0;              // kappaN/N
  double inv_rho_f64;
  float chi0[TYPES_MAX * TYPES_MAX];    // chi_ij N / N
  double chiN[TYPES_MAX * TYPES_MAX];   // chi_ij N
};
cudaError_t launch_fields_types(const TypesArgs& a, unsigned* arrive, int sm_count,
                                cudaStream_t st);
cudaError_t launch_histogram_types(const Geom& g, const float* x, const float* y, const float* z,
                                   const uint8_t* ttab, const uint8_t* mol_arch, uint32_t* n,
                                   int sm_count, cudaStream_t st);
// n_i | n_j << 16 per cell from the type planes n (for the composition S(q))
cudaError_t launch_pack_type_pair(const uint32_t* n, uint32_t cells, uint32_t ti, uint32_t tj,
                                  uint32_t* out, unsigned* err, int sm_count, cudaStream_t st);
// out[2] = sum over cells of the energy per cell, out[3] = largest total count,
// out[4] = 0 (no external potential); part: 2 * OBS_BLOCKS doubles
cudaError_t launch_observables_types(const TypesArgs& a, double kappaN, const uint32_t* n,
                                     double* part, double* out, cudaStream_t st);

// Entry-point helpers implemented in api.cu (messages go to soma_last_error).
}  // namespace soma
#include "../../include/soma.h"
namespace soma {
soma_status describe(const soma_system_desc* d, Geom* g);
soma_status report(soma_status st, const char* msg);
soma_status report_cuda(cudaError_t e, const char* what);
}  // namespace soma
