// grid.cu -- grid-side kernels of libsoma: the occupation count, the field
// update, the initial configuration and the FP64 observables.
//   - occupation numbers n_t(c): Eq. (density-characteristics), Sec. 3.1.1;
//   - fields omega_A/B: Eq. (omega-fields), option K^0;
//   - initial chains: Sec. 2.1 (Gaussian bonds, b0 = sqrt(3/k0));
//   - energies: Eq. (h-bond), (V-harmonic), (discrete-ham); S(q): Sec. 5.6.
#include "kernels.h"
#include "draws.cuh"
#include "omega.cuh"
#include "square_sum.cuh"

namespace soma {

// ---------------------------------------------------------------------------
// Occupation count of a whole configuration (used outside the sweep, whose
// epilogue counts on its own).  One thread per particle.
__global__ void histogram_kernel(const Geom g, const float* __restrict__ x,
                                 const float* __restrict__ y, const float* __restrict__ z,
                                 uint32_t* __restrict__ n, const uint64_t* __restrict__ seq,
                                 const uint8_t* __restrict__ arch,
                                 const uint8_t* __restrict__ alen) {
  const uint64_t M = g.n_chains * g.N;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t m = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; m < M; m += stride) {
    const uint64_t chain = m / g.N;
    const uint32_t i = (uint32_t)(m - chain * g.N);
    if (alen && i >= alen[arch[chain]]) continue;   // an absent slot
    const bool isB = seq ? ((seq[arch[chain]] >> i) & 1ull) != 0 : i >= g.N_A;
    atomicAdd(n + cell_of(g, x[m], y[m], z[m]), isB ? 0x10000u : 1u);
  }
}

cudaError_t launch_histogram(const Geom& g, const float* x, const float* y, const float* z,
                             uint32_t* n, int sm_count, cudaStream_t st, const uint64_t* seq,
                             const uint8_t* arch, const uint8_t* alen) {
  const uint64_t M = g.n_chains * g.N;
  uint64_t blocks = (M + 255) / 256;
  const uint64_t cap = (uint64_t)sm_count * 8;
  if (blocks > cap) blocks = cap;
  histogram_kernel<<<(unsigned)blocks, 256, 0, st>>>(g, x, y, z, n, seq, arch, alen);
  return cudaGetLastError();
}

// Range check of positions given by the caller: flag = 1 if any value is not
// finite or has |v| >= lim (the supported range of the cell fold).
// p starts 16-byte aligned (every position plane is 256-byte aligned): four
// coordinates per 16-byte load, the last n mod 4 one by one.
__global__ void __launch_bounds__(256) range_check_kernel(const float* __restrict__ p, uint64_t n,
                                                          float lim, unsigned* flag) {
  unsigned bad = 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t n4 = n / 4;
  const float4* __restrict__ q = reinterpret_cast<const float4*>(p);
  for (uint64_t i = tid; i < n4; i += stride) {
    const float4 v = __ldg(q + i);
    bad |= !(fabsf(v.x) < lim) | !(fabsf(v.y) < lim) | !(fabsf(v.z) < lim) | !(fabsf(v.w) < lim);
  }
  for (uint64_t i = 4 * n4 + tid; i < n; i += stride) bad |= !(fabsf(p[i]) < lim);
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1u);
}

// Copies the three planes of a caller's positions (src + d n) into the handle's
// (dst + d plane) and checks their range on the way: one launch and one read
// of the positions where three copies and three checks took two reads of them
// (analysis of a 16.8M-particle melt 554 -> 507 us).  VEC: the source planes are 16-byte aligned
// (n a multiple of 4); the destination's always are.
template <bool VEC>
__global__ void __launch_bounds__(256) copy_check_kernel(const float* __restrict__ src,
                                                         float* __restrict__ dst, uint64_t n,
                                                         uint64_t plane, float lim, unsigned* flag) {
  unsigned bad = 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const float* __restrict__ s = src + blockIdx.y * n;
  float* __restrict__ d = dst + blockIdx.y * plane;
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (VEC) {
    const uint64_t n4 = n / 4;
    for (; i < n4; i += stride) {
      const float4 v = __ldcs(reinterpret_cast<const float4*>(s) + i);
      bad |= !(fabsf(v.x) < lim) | !(fabsf(v.y) < lim) | !(fabsf(v.z) < lim) | !(fabsf(v.w) < lim);
      reinterpret_cast<float4*>(d)[i] = v;
    }
  } else {
    for (; i < n; i += stride) {
      const float v = __ldcs(s + i);
      bad |= !(fabsf(v) < lim);
      d[i] = v;
    }
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1u);
}

cudaError_t launch_copy_check(const float* src, float* dst, uint64_t n, uint64_t plane, float lim,
                              unsigned* flag, int sm_count, cudaStream_t st) {
  const bool vec = n % 4 == 0 && (reinterpret_cast<uintptr_t>(src) & 15u) == 0;
  uint64_t blocks = ((vec ? n / 4 : n) + 255) / 256;
  const uint64_t cap = (uint64_t)sm_count * 4;
  if (blocks > cap) blocks = cap;
  const dim3 grid((unsigned)blocks, 3);
  if (vec) copy_check_kernel<true><<<grid, 256, 0, st>>>(src, dst, n, plane, lim, flag);
  else copy_check_kernel<false><<<grid, 256, 0, st>>>(src, dst, n, plane, lim, flag);
  return cudaGetLastError();
}

cudaError_t launch_range_check(const float* p, uint64_t n, float lim, unsigned* flag, int sm_count,
                               cudaStream_t st) {
  uint64_t blocks = (n / 4 + 255) / 256;
  const uint64_t cap = (uint64_t)sm_count * 8;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  range_check_kernel<<<(unsigned)blocks, 256, 0, st>>>(p, n, lim, flag);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Field update: omega from the packed counts of one buffer, while the other
// buffer is cleared for the next sweep's count.  The last block to finish
// (arrival counter, no waiting) advances the sweep counter, so every block
// read the same counter value.
//
// TAB: the table of a smart Monte Carlo or tensor-core learned sweep in the same
// pass.  Per type and cell, one entry a move reads with 16-byte loads instead of
// gathering seven field values:
//   FIELD_FORCE: omega and minus its central difference along each axis
//     (float4, A plane then B plane);
//   FIELD_GRADIENT: omega, its three lower face differences, and the
//     differences of the upper and lower ones (two float4).
// The neighbours' omega are evaluated from their counts (the bits that are
// stored for them), so the table needs no second kernel behind this one and no
// second read of the planes: 2.1M particles of N = 33, 20 cycles 849 -> 820 us.
//
// PLAIN: K^0 without external fields, the usual case, whose omega then costs no
// branches; a thread's cell coordinates advance by a fixed step instead of two
// divisions per cell.
template <typename WT, int TAB, bool PLAIN>
__global__ void __launch_bounds__(256) fields_kernel(const FieldArgs p, unsigned* arrive) {
  chained_begin();
  const unsigned long long s = *p.d_sweep;
  const int rd = p.after_sweep ? (int)((s + 1ull) & 1ull) : (int)(s & 1ull);
  const uint32_t* __restrict__ nr = rd ? p.n1 : p.n0;
  uint32_t* __restrict__ nc = rd ? p.n0 : p.n1;
  WT* __restrict__ wA = static_cast<WT*>(p.wA);
  WT* __restrict__ wB = static_cast<WT*>(p.wB);
  unsigned bad = 0;
  const uint32_t stride = gridDim.x * blockDim.x;
  const uint32_t nx = p.g.nx, ny = p.g.ny, nz = p.g.nz;
  uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t cx = 0, cy = 0, cz = 0, sx = 0, sy = 0, sz = 0;   // coordinates of c and of the stride
  if (TAB != FIELD_ONLY) {
    cx = c % nx;
    cy = (c / nx) % ny;
    cz = c / (nx * ny);
    sx = stride % nx;
    sy = (stride / nx) % ny;
    sz = stride / (nx * ny);
  }
  auto omega = [&](uint32_t v, uint32_t at, bool B) {
    return PLAIN ? load_cvt<WT>(store_cvt<WT>(omega_of(v, B, p.inv_rho, p.kappa0, p.half_chi0, 0)))
                 : omega_stored<WT>(p, v, at, B);
  };
  for (; c < p.g.cells; c += stride) {
    const uint32_t v = nr[c];
    nc[c] = 0u;
    const uint32_t a = v & 0xFFFFu, b = v >> 16;
    const float wa = omega(v, c, false), wb = omega(v, c, true);
    wA[c] = store_cvt<WT>(wa);
    wB[c] = store_cvt<WT>(wb);
    bad |= (a >= 0xC000u) | (b >= 0xC000u);
    if (TAB != FIELD_ONLY) {
      const uint32_t at[6] = {cx == 0 ? c + nx - 1 : c - 1,
                              cx + 1 == nx ? c + 1 - nx : c + 1,
                              cy == 0 ? c + (ny - 1) * nx : c - nx,
                              cy + 1 == ny ? c - (ny - 1) * nx : c + nx,
                              cz == 0 ? c + (nz - 1) * ny * nx : c - ny * nx,
                              cz + 1 == nz ? c - (nz - 1) * ny * nx : c + ny * nx};
      uint32_t u[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) u[k] = nr[at[k]];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const float w0 = t ? wb : wa;
        float w[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) w[k] = omega(u[k], at[k], t != 0);
        if (TAB == FIELD_FORCE) {
          p.tab[t * p.g.cells + c] =
              make_float4(w0, -0.5f * (w[1] - w[0]), -0.5f * (w[3] - w[2]), -0.5f * (w[5] - w[4]));
        } else {
          const float lo0 = w0 - w[0], lo1 = w0 - w[2], lo2 = w0 - w[4];
          float4* e = p.tab + 2u * ((size_t)t * p.g.cells + c);
          e[0] = make_float4(w0, lo0, lo1, lo2);
          e[1] = make_float4((w[1] - w0) - lo0, (w[3] - w0) - lo1, (w[5] - w0) - lo2, 0.f);
        }
      }
      cx += sx;
      cy += sy;
      cz += sz;
      if (cx >= nx) { cx -= nx; ++cy; }
      if (cy >= ny) { cy -= ny; ++cz; }
    }
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(p.err, ERR_OVERFLOW);
  if (p.after_sweep && threadIdx.x == 0) {
    __threadfence();
    const unsigned done = atomicAdd(arrive, 1u);
    if (done == gridDim.x - 1) {
      *arrive = 0u;
      *p.d_sweep = s + 1ull;
    }
  }
}

template <typename WT, bool PLAIN>
static const void* fields_ptr_of(int tab_kind) {
  return tab_kind == FIELD_FORCE      ? (const void*)fields_kernel<WT, FIELD_FORCE, PLAIN>
         : tab_kind == FIELD_GRADIENT ? (const void*)fields_kernel<WT, FIELD_GRADIENT, PLAIN>
                                      : (const void*)fields_kernel<WT, FIELD_ONLY, PLAIN>;
}
template <typename WT>
static const void* fields_ptr(int tab_kind, bool plain) {
  return plain ? fields_ptr_of<WT, true>(tab_kind) : fields_ptr_of<WT, false>(tab_kind);
}

cudaError_t launch_fields(const FieldArgs& a, unsigned* arrive, int grid_dtype, int sm_count,
                          cudaStream_t st) {
  uint64_t blocks = ((uint64_t)a.g.cells + 255) / 256;
  const uint64_t cap = (uint64_t)sm_count * 8;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  const int kind = a.tab ? a.tab_kind : FIELD_ONLY;
  const bool plain = a.hamiltonian == 0 && !a.ext && !a.forbidden;
  const void* fn = grid_dtype == 1   ? fields_ptr<__nv_bfloat16>(kind, plain)
                   : grid_dtype == 2 ? fields_ptr<__half>(kind, plain)
                                     : fields_ptr<float>(kind, plain);
  void* args[] = {const_cast<FieldArgs*>(&a), &arrive};
  return launch_chained(fn, dim3((unsigned)blocks), dim3(256), args, 0, st);
}

template <typename WT>
__global__ void convert_kernel(const WT* __restrict__ w, float* __restrict__ dst, uint64_t n) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    dst[i] = load_w<WT>(w, (uint32_t)i);
}

cudaError_t launch_convert_fields(const void* w, int grid_dtype, float* dst, uint64_t n,
                                  cudaStream_t st) {
  const unsigned blocks = 1024;
  switch (grid_dtype) {
    case 1: convert_kernel<<<blocks, 256, 0, st>>>((const __nv_bfloat16*)w, dst, n); break;
    case 2: convert_kernel<<<blocks, 256, 0, st>>>((const __half*)w, dst, n); break;
    default: convert_kernel<<<blocks, 256, 0, st>>>((const float*)w, dst, n); break;
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Initial configuration, one thread per chain, FP64 with explicit rounding
// (no contraction) so the arithmetic is the textbook one: first particle
// uniform in the box, then N-1 bond vectors with components sigma * z, z from
// the Box-Muller transform of two open uniforms.
__global__ void init_kernel(const Geom g, float* __restrict__ x, float* __restrict__ y,
                            float* __restrict__ z, double sigma) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint32_t ctr3 = (PURPOSE_INIT << 24) | (g.replica & 0xFFFFFFu);
  const double two_pi = 6.283185307179586;  // 2*pi rounded to FP64
  for (uint64_t chain = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; chain < g.n_chains;
       chain += stride) {
    const uint64_t gc = chain + g.chain_base;   // the chain's index in the whole system
    const uint32_t lo = (uint32_t)gc, hi = (uint32_t)(gc >> 32);
    uint4 w = philox4x32_10(make_uint4(lo, hi, 0u, ctr3), g.key0, g.key1);
    double r[3] = {__dmul_rn(uniform_open_f64(w.x), (double)g.nx),
                   __dmul_rn(uniform_open_f64(w.y), (double)g.ny),
                   __dmul_rn(uniform_open_f64(w.z), (double)g.nz)};
    const uint64_t m0 = chain * g.N;
    x[m0] = (float)r[0];
    y[m0] = (float)r[1];
    z[m0] = (float)r[2];
    uint32_t cached = 0xFFFFFFFFu;
    for (uint32_t i = 0; i + 1 < g.N; ++i) {
      for (int d = 0; d < 3; ++d) {
        const uint32_t j = 3u * i + (uint32_t)d;
        const uint32_t call = 1u + j / 4u;
        if (call != cached) {
          w = philox4x32_10(make_uint4(lo, hi, call, ctr3), g.key0, g.key1);
          cached = call;
        }
        const uint32_t pr = (j % 4u) / 2u;
        const double u1 = uniform_open_f64(pr ? w.z : w.x);
        const double u2 = uniform_open_f64(pr ? w.w : w.y);
        const double rad = sqrt(__dmul_rn(-2.0, log(u1)));
        const double th = __dmul_rn(two_pi, u2);
        const double gz = (j % 2u == 0u) ? __dmul_rn(rad, cos(th)) : __dmul_rn(rad, sin(th));
        r[d] = __dadd_rn(r[d], __dmul_rn(sigma, gz));
      }
      x[m0 + i + 1] = (float)r[0];
      y[m0 + i + 1] = (float)r[1];
      z[m0 + i + 1] = (float)r[2];
    }
  }
}

cudaError_t launch_init(const Geom& g, float* x, float* y, float* z, double sigma, int sm_count,
                        cudaStream_t st) {
  uint64_t blocks = (g.n_chains + 127) / 128;
  const uint64_t cap = (uint64_t)sm_count * 16;
  if (blocks > cap) blocks = cap;
  init_kernel<<<(unsigned)blocks, 128, 0, st>>>(g, x, y, z, sigma);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Spatial labelling of chains at initialisation: key = Morton code of the
// 8^3-cell block of the chain's first particle, packed above the old label so
// all keys are distinct and the sorted order is unique; a bitonic network
// sorts them; a gather moves whole chains to their new labels.
constexpr uint32_t SORT_BLOCK_SHIFT = 3;  // 8-cell blocks

__global__ void chain_key_kernel(const Geom g, const float* __restrict__ x,
                                 const float* __restrict__ y, const float* __restrict__ z,
                                 uint64_t* __restrict__ keys, uint64_t n_pad) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_pad; k += stride) {
    if (k >= g.n_chains) {
      keys[k] = ~0ull;
      continue;
    }
    const uint64_t m = k * g.N;
    const uint32_t b[3] = {
        fold_axis(g, 0, x[m], (uint32_t)g.nx) >> SORT_BLOCK_SHIFT,
        fold_axis(g, 1, y[m], (uint32_t)g.ny) >> SORT_BLOCK_SHIFT,
        fold_axis(g, 2, z[m], (uint32_t)g.nz) >> SORT_BLOCK_SHIFT};
    uint64_t key = 0;
    for (int bit = 0; bit < 10; ++bit)
      for (int d = 0; d < 3; ++d) key |= (uint64_t)((b[d] >> bit) & 1u) << (3 * bit + d);
    keys[k] = (key << 32) | k;
  }
}

__global__ void bitonic_step_kernel(uint64_t* __restrict__ a, uint64_t n, uint64_t j, uint64_t k) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const uint64_t l = i ^ j;
    if (l <= i) continue;
    const uint64_t u = a[i], v = a[l];
    const bool up = (i & k) == 0;
    if ((u > v) == up) {
      a[i] = v;
      a[l] = u;
    }
  }
}

__global__ void chain_gather_kernel(const Geom g, const uint64_t* __restrict__ keys,
                                    const float* __restrict__ src, float* __restrict__ dst,
                                    uint64_t src_plane, uint64_t dst_plane) {
  const uint64_t M = g.n_chains * g.N;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t m = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; m < M; m += stride) {
    const uint64_t j = m / g.N, i = m - j * g.N;
    const uint64_t old = keys[j] & 0xFFFFFFFFull;
    const uint64_t from = old * g.N + i;
#pragma unroll
    for (int d = 0; d < 3; ++d) dst[d * dst_plane + m] = src[d * src_plane + from];
  }
}

cudaError_t launch_sort_chains(const Geom& g, const float* src, uint64_t src_plane, float* dst,
                               uint64_t dst_plane, uint64_t* keys, uint64_t n_pad, int sm_count,
                               cudaStream_t st) {
  const unsigned blocks = (unsigned)sm_count * 8;
  chain_key_kernel<<<blocks, 256, 0, st>>>(g, src, src + src_plane, src + 2 * src_plane, keys,
                                           n_pad);
  for (uint64_t k = 2; k <= n_pad; k <<= 1)
    for (uint64_t j = k >> 1; j > 0; j >>= 1)
      bitonic_step_kernel<<<blocks, 256, 0, st>>>(keys, n_pad, j, k);
  chain_gather_kernel<<<blocks, 256, 0, st>>>(g, keys, src, dst, src_plane, dst_plane);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Sums over bonds |b|^2 and over chains |R_e|^2 (square_sum.cuh).
//
// One thread per particle; the positions are read once from memory (a bond's
// upper particle hits the line of the next lane).  With the squares in FP64 the
// kernel was bound by that pipe (two lanes per SM and cycle, 87 % busy, and the
// one chain end in a warp cost it a whole warp's operations): 748 us for 16.8M
// particles.  With the kernels below the analysis of that melt (64 wave
// vectors) went from 1.48 to 0.57 ms.
__global__ void __launch_bounds__(256) chain_obs_kernel(const Geom g, const float* __restrict__ x,
                                                        const float* __restrict__ y,
                                                        const float* __restrict__ z,
                                                        double* __restrict__ part) {
  __shared__ double sh[2 * 32];
  const uint64_t M = g.n_chains * g.N;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint32_t N = g.N, step = (uint32_t)(stride % N);
  uint64_t m = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t i = (uint32_t)(m % N);
  SquareSum bonds, ends;
  for (; m < M; m += stride) {
    const float x0 = x[m], y0 = y[m], z0 = z[m];
    if (i + 1u < N) bonds.add(x[m + 1], y[m + 1], z[m + 1], x0, y0, z0);
    if (i == 0u) {
      const uint64_t e = m + N - 1u;
      ends.add(x[e], y[e], z[e], x0, y0, z0);
    }
    i += step;
    if (i >= N) i -= N;
  }
  double v[2] = {bonds.value(), ends.value()};
  block_sum<2>(v, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x * 2 + 0] = v[0];
    part[blockIdx.x * 2 + 1] = v[1];
  }
}

// Energy of the occupation numbers.  With rho = rho_0 dL^3, r = round(rho) and
// the integers d = n_A + n_B - r and f = n_A - n_B, a cell's energy is
//   kappaN/2 (d + r - rho)^2/rho^2 - chiN/4 f^2/rho^2     (K^0; K^1: + chiN n_A n_B/rho^2),
// so the sums of d, d^2 and f^2 (or n_A n_B) over a block's cells are taken as
// exact integers and combined in FP64 once per block: no FP64 operation per
// cell (39 us before at 96^3 cells), and the squares of the deviations are
// summed without cancellation.  The external energy, if any, is summed in FP64.
__global__ void __launch_bounds__(256) grid_obs_kernel(const Geom g, const uint32_t* __restrict__ n,
                                                       double inv_rho, double kappaN, double chiN,
                                                       int hamiltonian, const float* __restrict__ ext,
                                                       double* __restrict__ part) {
  __shared__ double sh[32];
  __shared__ long long si[3][8];
  __shared__ uint32_t sm[2][8];
  const double rho = 1.0 / inv_rho;
  const long long r = llrint(rho < 131072.0 ? rho : 131072.0);   // counts stay below 2^17
  long long s1 = 0, s2 = 0, s3 = 0;
  uint32_t mx = 0u, cnt = 0u;
  double e_ext[1] = {0.0};
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < g.cells; c += stride) {
    const uint32_t w = n[c];
    const uint32_t a = w & 0xFFFFu, b = w >> 16;
    const int d = (int)(a + b) - (int)r, f = (int)a - (int)b;
    s1 += d;
    s2 += (long long)d * d;
    s3 += hamiltonian ? (long long)a * b : (long long)f * f;
    mx = max(mx, a + b);
    ++cnt;
    if (ext) e_ext[0] += (double)a * (double)ext[c] + (double)b * (double)ext[g.cells + c];
  }
  for (int o = 16; o > 0; o >>= 1) {
    s1 += __shfl_xor_sync(FULL, s1, o);
    s2 += __shfl_xor_sync(FULL, s2, o);
    s3 += __shfl_xor_sync(FULL, s3, o);
    mx = max(mx, __shfl_xor_sync(FULL, mx, o));
    cnt += __shfl_xor_sync(FULL, cnt, o);
  }
  if ((threadIdx.x & 31) == 0) {
    const int k = threadIdx.x >> 5;
    si[0][k] = s1;
    si[1][k] = s2;
    si[2][k] = s3;
    sm[0][k] = mx;
    sm[1][k] = cnt;
  }
  if (ext) block_sum<1>(e_ext, sh);   // uniform: ext is a kernel argument
  __syncthreads();
  if (threadIdx.x == 0) {
    s1 = s2 = s3 = 0;
    mx = cnt = 0u;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
      s1 += si[0][k];
      s2 += si[1][k];
      s3 += si[2][k];
      mx = max(mx, sm[0][k]);
      cnt += sm[1][k];
    }
    const double off = (double)r - rho;
    const double fl = (double)s2 + off * (2.0 * (double)s1 + off * (double)cnt);
    const double K = inv_rho * inv_rho *
                     (0.5 * kappaN * fl + (hamiltonian ? chiN : -0.25 * chiN) * (double)s3);
    part[2 * OBS_BLOCKS + blockIdx.x * 3 + 0] = K;
    part[2 * OBS_BLOCKS + blockIdx.x * 3 + 1] = (double)mx;
    part[2 * OBS_BLOCKS + blockIdx.x * 3 + 2] = e_ext[0];
  }
}

// Folds the blocks' sums in a fixed order, one block of threads instead of one
// thread (306 us before with 1024 blocks each, the FP64 additions and their
// loads one after another).
__global__ void __launch_bounds__(256) obs_final_kernel(const double* __restrict__ part, int nb_chain,
                                                        int nb_grid, double* __restrict__ out) {
  __shared__ double sh[4 * 32];
  __shared__ double shm[8];
  double v[4] = {0.0, 0.0, 0.0, 0.0}, mx = 0.0;
  for (int i = threadIdx.x; i < nb_chain; i += 256) {
    v[0] += part[2 * i];
    v[1] += part[2 * i + 1];
  }
  for (int i = threadIdx.x; i < nb_grid; i += 256) {
    v[2] += part[2 * OBS_BLOCKS + 3 * i];
    mx = fmax(mx, part[2 * OBS_BLOCKS + 3 * i + 1]);
    v[3] += part[2 * OBS_BLOCKS + 3 * i + 2];
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(FULL, mx, o));
  if ((threadIdx.x & 31) == 0) shm[threadIdx.x >> 5] = mx;
  block_sum<4>(v, sh);
  if (threadIdx.x != 0) return;
  for (int k = 1; k < 8; ++k) mx = fmax(mx, shm[k]);
  out[0] = v[0];
  out[1] = v[1];
  out[2] = v[2];
  out[3] = mx;
  out[4] = v[3];
}

cudaError_t launch_observables(const Geom& g, const float* x, const float* y, const float* z,
                               const uint32_t* n, double inv_rho, double kappaN, double chiN,
                               int hamiltonian, const float* ext, double* part, double* out,
                               cudaStream_t st) {
  const uint64_t M = g.n_chains * g.N;
  uint64_t nb1 = (M + 255) / 256;
  if (nb1 > OBS_BLOCKS) nb1 = OBS_BLOCKS;
  uint64_t nb2 = ((uint64_t)g.cells + 255) / 256;
  if (nb2 > OBS_BLOCKS) nb2 = OBS_BLOCKS;
  chain_obs_kernel<<<(unsigned)nb1, 256, 0, st>>>(g, x, y, z, part);
  grid_obs_kernel<<<(unsigned)nb2, 256, 0, st>>>(g, n, inv_rho, kappaN, chiN, hamiltonian, ext,
                                                 part);
  obs_final_kernel<<<1, 256, 0, st>>>(part, (int)nb1, (int)nb2, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// S(q) = |sum_c dn(c) e^{-i q.c}|^2 / M with e^{-i q.c} the product of three
// per-axis twiddles, entries of one FP64 table per axis (e^{-2 pi i r/n}, r < n).
//
// FP64 arithmetic bounds it (this chip issues two FP64 lanes per SM and cycle),
// so the sum is taken axis by axis, the x axis of a row once for every distinct
// |q_x| instead of once per wave vector: with dn real, cells x and n - x share
// a cosine and a sine, so a row costs one FP64 multiply-add per cell and
// distinct |q_x| (their sum and difference are integers), then eight per wave
// vector.  The direct triple product took ten operations per cell and wave
// vector.  A block takes R = 256/DP rows at a time (DP: the distinct |q_x|
// rounded up to a power of two from 4 to 32), thread (row, distinct q_x) sums
// along x over chunks staged in shared memory, then thread (q, row mod 8)
// multiplies in the y and z twiddles.  The analysis of a 16.8M-particle melt
// (96^3 cells, 64 wave vectors) went from 3.19 to 1.48 ms.
constexpr int SQ_CHUNK = 32;

struct SqWaves {
  int k, distinct;
  uint16_t my[SQ_MAX], mz[SQ_MAX];   // reduced into [0, n)
  uint16_t mx[SQ_MAX];               // the distinct |m_x|, reduced into [0, n/2]
  uint8_t dx[SQ_MAX];                // which of them wave vector q has
  uint8_t conj[SQ_MAX];              // q_x is the negative of that one
};

template <int DP>
__global__ void __launch_bounds__(256) sq_kernel(const Geom g, const uint32_t* __restrict__ n,
                                                 const double2* __restrict__ tw, const SqWaves w,
                                                 double* __restrict__ part) {
  constexpr int R = 256 / DP;
  __shared__ double2 eo[R][SQ_CHUNK + 1];   // sum and difference of cells x and n - x
  __shared__ double2 xs[R][DP + 1];         // the rows' sums along x
  __shared__ double2 red[8][SQ_MAX];
  const uint32_t nx = g.nx, ny = g.ny, nz = g.nz, rows = ny * nz, half = nx / 2u + 1u;
  const int t = threadIdx.x, r = t / DP, d = t % DP;
  const int q = t & 31, grp = t >> 5;
  const uint32_t mf = d < w.distinct ? w.mx[d] : 0u;
  double re = 0.0, im = 0.0;
  for (uint32_t row0 = blockIdx.x * R; row0 < rows; row0 += gridDim.x * R) {
    double C = 0.0, S = 0.0;
    uint32_t idx = 0;
    for (uint32_t x0 = 0; x0 < half; x0 += SQ_CHUNK) {
      __syncthreads();
      for (int p = t; p < R * SQ_CHUNK; p += 256) {
        const uint32_t row = row0 + p / SQ_CHUNK, x = x0 + p % SQ_CHUNK;
        int e = 0, o = 0;
        if (row < rows && x < half) {
          const uint32_t* line = n + (size_t)row * nx;
          const uint32_t v = __ldg(line + x);
          e = (int)(v & 0xFFFFu) - (int)(v >> 16);
          const uint32_t x2 = nx - x;
          if (x != 0u && x2 != x) {
            const uint32_t u = __ldg(line + x2);
            const int f = (int)(u & 0xFFFFu) - (int)(u >> 16);
            o = e - f;
            e += f;
          }
        }
        eo[p / SQ_CHUNK][p % SQ_CHUNK] = make_double2((double)e, (double)o);
      }
      __syncthreads();
      if (d < w.distinct) {
        const int m = (int)min((uint32_t)SQ_CHUNK, half - x0);
#pragma unroll 4
        for (int x = 0; x < m; ++x) {
          const double2 c = __ldg(tw + idx);
          const double2 v = eo[r][x];
          idx += mf;
          if (idx >= nx) idx -= nx;
          C = fma(v.x, c.x, C);
          S = fma(v.y, c.y, S);
        }
      }
    }
    if (d < w.distinct) xs[r][d] = make_double2(C, S);
    __syncthreads();
    if (q < w.k) {
      for (int rr = grp; rr < R && row0 + rr < rows; rr += 8) {
        const uint32_t row = row0 + rr, z = row / ny, y = row - z * ny;
        const double2 a = __ldg(tw + nx + (w.my[q] * y) % ny);
        const double2 b = __ldg(tw + nx + ny + (w.mz[q] * z) % nz);
        const double2 v = xs[rr][w.dx[q]];
        const double vi = w.conj[q] ? -v.y : v.y;
        const double pr = a.x * b.x - a.y * b.y, pi = a.x * b.y + a.y * b.x;
        re += v.x * pr - vi * pi;
        im += v.x * pi + vi * pr;
      }
    }
  }
  red[grp][q] = make_double2(re, im);
  __syncthreads();
  if (grp == 0 && q < w.k) {
    for (int k = 1; k < 8; ++k) {
      re += red[k][q].x;
      im += red[k][q].y;
    }
    part[blockIdx.x * 2 * SQ_MAX + 2 * q] = re;
    part[blockIdx.x * 2 * SQ_MAX + 2 * q + 1] = im;
  }
}

// One warp per wave vector folds the blocks' sums in a fixed order, four warps
// to a block (one block for all took 13 us on one SM's FP64 pipe).
__global__ void __launch_bounds__(128) sq_final_kernel(const double* __restrict__ part, int nb,
                                                               int k, double invM,
                                                               double* __restrict__ out) {
  const int q = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (q >= k) return;
  double re = 0.0, im = 0.0;
  for (int b = lane; b < nb; b += 32) {
    const double2 v = reinterpret_cast<const double2*>(part)[b * SQ_MAX + q];
    re += v.x;
    im += v.y;
  }
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_xor_sync(FULL, re, o);
    im += __shfl_xor_sync(FULL, im, o);
  }
  if (lane == 0) out[q] = (re * re + im * im) * invM;
}

cudaError_t launch_structure_factor(const Geom& g, const uint32_t* n, const double* tw,
                                    const int32_t* m, int k, double* part, double* out,
                                    cudaStream_t st) {
  SqWaves w = {};
  w.k = k;
  for (int q = 0; q < k; ++q) {
    const int64_t rx = (((int64_t)m[3 * q] % g.nx) + g.nx) % g.nx;
    const int64_t mf = rx <= g.nx - rx ? rx : g.nx - rx;
    w.conj[q] = mf != rx;
    w.my[q] = (uint16_t)((((int64_t)m[3 * q + 1] % g.ny) + g.ny) % g.ny);
    w.mz[q] = (uint16_t)((((int64_t)m[3 * q + 2] % g.nz) + g.nz) % g.nz);
    int d = 0;
    while (d < w.distinct && w.mx[d] != mf) ++d;
    if (d == w.distinct) w.mx[w.distinct++] = (uint16_t)mf;
    w.dx[q] = (uint8_t)d;
  }
  const int dp = w.distinct <= 4 ? 4 : w.distinct <= 8 ? 8 : w.distinct <= 16 ? 16 : 32;
  const uint64_t per = 256u / (unsigned)dp;
  uint64_t nb = ((uint64_t)g.ny * g.nz + per - 1) / per;
  if (nb > SQ_BLOCKS) nb = SQ_BLOCKS;
  const double2* tw2 = reinterpret_cast<const double2*>(tw);
  switch (dp) {
    case 4: sq_kernel<4><<<(unsigned)nb, 256, 0, st>>>(g, n, tw2, w, part); break;
    case 8: sq_kernel<8><<<(unsigned)nb, 256, 0, st>>>(g, n, tw2, w, part); break;
    case 16: sq_kernel<16><<<(unsigned)nb, 256, 0, st>>>(g, n, tw2, w, part); break;
    default: sq_kernel<32><<<(unsigned)nb, 256, 0, st>>>(g, n, tw2, w, part); break;
  }
  const double invM = 1.0 / (double)g.particles;
  sq_final_kernel<<<(k + 3) / 4, 128, 0, st>>>(part, (int)nb, k, invM, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
__global__ void philox_kernel(const uint32_t* __restrict__ ctr, const uint32_t* __restrict__ key,
                              uint32_t* __restrict__ out, size_t n) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
  const uint4 r = philox4x32_10(c, key[2 * i], key[2 * i + 1]);
  out[4 * i] = r.x;
  out[4 * i + 1] = r.y;
  out[4 * i + 2] = r.z;
  out[4 * i + 3] = r.w;
}

cudaError_t launch_philox(const uint32_t* ctr, const uint32_t* key, uint32_t* out, size_t n,
                          cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  philox_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(ctr, key, out, n);
  return cudaGetLastError();
}

// What a smart Monte Carlo move makes of its draw (four words): the three
// normals and ln u of the spare 24 bits, by the sweeps' own device functions.
__global__ void smc_draws_kernel(const uint32_t* __restrict__ w, float* __restrict__ out,
                                 size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const uint4 r = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
    float gx, gy, gz;
    smc_normals(r, gx, gy, gz);
    out[4 * i] = gx;
    out[4 * i + 1] = gy;
    out[4 * i + 2] = gz;
    out[4 * i + 3] = log_uniform_open(spare_uniform_word(r));
  }
}

cudaError_t launch_smc_draws(const uint32_t* words, float* out, size_t n, int sm_count,
                             cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const size_t blocks = (n + 255) / 256;
  const size_t cap = (size_t)8 * (size_t)(sm_count > 0 ? sm_count : 1);
  smc_draws_kernel<<<(unsigned)(blocks < cap ? blocks : cap), 256, 0, st>>>(words, out, n);
  return cudaGetLastError();
}

}  // namespace soma
