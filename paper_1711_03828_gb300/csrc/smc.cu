// smc.cu -- the smart Monte Carlo (force-biased) sweep kernels.
//
// Trial move dr = A F(r) + sqrt(2A) xi with A = a^2/6, F the bonded force
// minus the central-difference gradient of omega_t over the six neighbouring
// cells, accepted with min(1, exp(-dE) T(r'->r)/T(r->r')) (Sec. 2.2 names the
// force-biased proposal; the Rossky-Doll-Friedman form is used).  One Philox
// draw per move (purpose 1): normals by Box-Muller from the top 24 bits of its
// four words, the acceptance uniform from the 24 bits they leave (the low
// bytes of words 0-2).  The radius sqrt(-2 ln u) takes ln u accurate to about an
// ulp (near u = 1 a small absolute error of ln u would be a large one of the
// radius); the angle takes the hardware sincos (absolute error about 2^-21,
// below 1e-6 dL in the displacement) and the acceptance test the hardware log,
// as the uniform move does.  The move stays exact whatever the normals'
// rounding: the acceptance evaluates both proposal densities at the realised
// trial position.
#include "kernels.h"
#include "pair_body.cuh"
#include "strip.cuh"
#include "draws.cuh"

namespace soma {

// ---------------------------------------------------------------------------
// Smart Monte Carlo step for even N <= 64 in the paired layout of
// pair_body.cuh: lane l holds the even particle 2l and the odd particle 2l+1
// of one chain; after the draws the pair is relabelled with the chain's
// set-order bit into A (moves in the first set) and B (second set), so that
// every lane moves one particle per set without divergent branches.  Trial
// move dr = A F(r) + sqrt(2A) xi, F = bonded force minus the central-difference
// gradient of omega_t over the six neighbouring cells; accepted with
// min(1, exp(-dE) T(r'->r)/T(r->r')), T(r->r') = exp(-|r'-r-A F(r)|^2/(4A)).
struct SmcSlot {
  float x, y, z;      // position
  float gx, gy, gz;   // standard normals
  float lnu;          // log of the acceptance uniform
  float w;            // omega at the old cell
  float fx, fy, fz;   // field force at the old cell
  uint32_t c;         // old cell
};

// The two slots of a lane, particles m and m + 1 of the draws' counters: the old
// cells' table entries first (in flight during the draws and normals).
__device__ __forceinline__ void smc_slots(const Geom& g, const float4* tab0, const float4* tab1,
                                          uint64_t m, uint32_t sweep, uint32_t ctr3a, SmcSlot& q0,
                                          SmcSlot& q1, uint32_t* first_word) {
  // an empty slot's cell lies in the grid; its values are not used
  q0.c = cell_of(g, q0.x, q0.y, q0.z);
  q1.c = cell_of(g, q1.x, q1.y, q1.z);
  q0.w = smc_field(tab0, q0.c, q0.fx, q0.fy, q0.fz);
  q1.w = smc_field(tab1, q1.c, q1.fx, q1.fy, q1.fz);
  const uint64_t m1 = m + 1u;
  const uint4 r0 = philox_rk(make_uint4((uint32_t)m, (uint32_t)(m >> 32), sweep, ctr3a), g);
  const uint4 r1 = philox_rk(make_uint4((uint32_t)m1, (uint32_t)(m1 >> 32), sweep, ctr3a), g);
  *first_word = r0.w;
  float n0[3], n1[3];
  smc_normals2(r0, r1, n0, n1);
  q0.gx = n0[0]; q0.gy = n0[1]; q0.gz = n0[2];
  q1.gx = n1[0]; q1.gy = n1[1]; q1.gz = n1[2];
  q0.lnu = log_uniform_open(spare_uniform_word(r0));
  q1.lnu = log_uniform_open(spare_uniform_word(r1));
}

// One smart Monte Carlo move of M against the fixed partner sum
// U = sum (r - n) over its k bonded partners; returns acceptance.
__device__ __forceinline__ bool smc_move(const SweepArgs& p, const float4* tab, SmcSlot& M, float ux,
                                         float uy, float uz, float k, bool valid) {
  const float A = p.smc_A, s2A = p.smc_s2A, K2 = 2.f * p.K_b;
  const float Fx = fmaf(-K2, ux, M.fx), Fy = fmaf(-K2, uy, M.fy), Fz = fmaf(-K2, uz, M.fz);
  const float tx = __fadd_rn(M.x, fmaf(s2A, M.gx, A * Fx));
  const float ty = __fadd_rn(M.y, fmaf(s2A, M.gy, A * Fy));
  const float tz = __fadd_rn(M.z, fmaf(s2A, M.gz, A * Fz));
  const uint32_t cn = cell_of(p.g, tx, ty, tz);
  float fnx, fny, fnz;
  const float w_new = smc_field(tab, cn, fnx, fny, fnz);
  const float dx = tx - M.x, dy = ty - M.y, dz = tz - M.z;
  const float du = fmaf(dx, ux, fmaf(dy, uy, dz * uz));
  const float dd = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
  const float dE = fmaf(p.K_b, fmaf(2.f, du, k * dd), w_new - M.w);
  const float Gx = fmaf(-K2, fmaf(k, dx, ux), fnx), Gy = fmaf(-K2, fmaf(k, dy, uy), fny),
              Gz = fmaf(-K2, fmaf(k, dz, uz), fnz);
  const float ax = dx - A * Fx, ay = dy - A * Fy, az = dz - A * Fz;
  const float bx = -dx - A * Gx, by = -dy - A * Gy, bz = -dz - A * Gz;
  const float fwd = fmaf(ax, ax, fmaf(ay, ay, az * az));
  const float rev = fmaf(bx, bx, fmaf(by, by, bz * bz));
  const float log_alpha = fmaf(fwd - rev, p.smc_inv4A, -dE);
  const bool acc = valid && (log_alpha >= 0.f || M.lnu < log_alpha);
  M.x = acc ? tx : M.x;
  M.y = acc ? ty : M.y;
  M.z = acc ? tz : M.z;
  M.c = acc ? cn : M.c;
  return acc;
}

// Paired smart Monte Carlo sweep (even N <= 64).  One block of 28 warps per
// SM (72 registers; 16 cycles of 67M particles with 24 warps 13.15 ms, 28 12.96, 32,
// with spills, 13.04) owns a contiguous range of tiles, which its warps take in order from a
// shared-memory counter, so all of them finish within a tile of each other.
__global__ void __launch_bounds__(896, 1) sweep_smc_pair_kernel(const SweepArgs p) {
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
  const uint32_t ctr3a = (PURPOSE_MOVE << 24) | (p.g.replica & 0xFFFFFFu);
  PairLane<float> L;
  L.init(lane, p.g.N, p.g.N_A, p.wA, p.wB);
  const float4* tab0 = p.smc_tab + (L.v0 == 1u ? 0u : p.g.cells);   // table plane of slot 0
  const float4* tab1 = p.smc_tab + (L.v1 == 1u ? 0u : p.g.cells);
  const uint32_t TN = p.G * p.g.N;
  const uint32_t dense_tiles = TN == 64u ? (uint32_t)p.full_tiles : 0u;   // all lanes hold a pair
  unsigned my_acc = 0;
  // positions of the warp's next tile, loaded while the current one is moved
  float2 nx = make_float2(0.f, 0.f), ny = nx, nz = nx;
  auto load_pos = [&](uint32_t t) {
    if (t < t_end && (t < dense_tiles || L.in_tile(t < (uint32_t)p.full_tiles, p.last_rows))) {
      const uint32_t b = t * TN + L.li0;
      nx = __ldcs(reinterpret_cast<const float2*>(p.x + b));
      ny = __ldcs(reinterpret_cast<const float2*>(p.y + b));
      nz = __ldcs(reinterpret_cast<const float2*>(p.z + b));
    }
  };
  uint32_t tile = claim();
  load_pos(tile);
  while (tile < t_end) {
    const bool valid = tile < dense_tiles || L.in_tile(tile < (uint32_t)p.full_tiles, p.last_rows);
    const uint32_t base = tile * TN + L.li0;
    float2 px = make_float2(0.f, 0.f), py = px, pz = px;
    if (valid) {
      px = nx;
      py = ny;
      pz = nz;
    }
    const uint32_t next_tile = claim();
    load_pos(next_tile);
    uint32_t w0;
    const uint32_t cbase = base + (uint32_t)p.g.id_base;
    SmcSlot s0, s1;
    s0.x = px.x; s0.y = py.x; s0.z = pz.x;
    s1.x = px.y; s1.y = py.y; s1.z = pz.y;
    smc_slots(p.g, tab0, tab1, cbase, sweep, ctr3a, s0, s1, &w0);
    const bool sw = p.set_order_random && (__shfl_sync(FULL, w0, L.first_lane) & 1u);
    SmcSlot A = sw ? s1 : s0, B = sw ? s0 : s1;
    const float4* tA = sw ? tab1 : tab0;
    const float4* tB = sw ? tab0 : tab1;
    {  // first set: A moves against B and the adjacent lane's B
      const int src = sw ? L.src_next : L.src_prev;
      const float cf = sw ? L.cf_next1 : L.cf_prev0;
      const float sx = __shfl_sync(FULL, B.x, src);
      const float sy = __shfl_sync(FULL, B.y, src);
      const float sz = __shfl_sync(FULL, B.z, src);
      my_acc += smc_move(p, tA, A, fmaf(cf, A.x - sx, A.x - B.x), fmaf(cf, A.y - sy, A.y - B.y),
                             fmaf(cf, A.z - sz, A.z - B.z), 1.f + cf, valid);
    }
    {  // second set: B moves against A and the adjacent lane's A
      const int src = sw ? L.src_prev : L.src_next;
      const float cf = sw ? L.cf_prev0 : L.cf_next1;
      const float sx = __shfl_sync(FULL, A.x, src);
      const float sy = __shfl_sync(FULL, A.y, src);
      const float sz = __shfl_sync(FULL, A.z, src);
      my_acc += smc_move(p, tB, B, fmaf(cf, B.x - sx, B.x - A.x), fmaf(cf, B.y - sy, B.y - A.y),
                             fmaf(cf, B.z - sz, B.z - A.z), 1.f + cf, valid);
    }
    if (valid) {
      __stcs(reinterpret_cast<float2*>(p.x + base), sw ? make_float2(B.x, A.x) : make_float2(A.x, B.x));
      __stcs(reinterpret_cast<float2*>(p.y + base), sw ? make_float2(B.y, A.y) : make_float2(A.y, B.y));
      __stcs(reinterpret_cast<float2*>(p.z + base), sw ? make_float2(B.z, A.z) : make_float2(A.z, B.z));
      const uint32_t vA = sw ? L.v1 : L.v0, vB = sw ? L.v0 : L.v1;
      const bool same = A.c == B.c;
      atomicAdd(nacc + A.c, same ? vA + vB : vA);
      if (!same) atomicAdd(nacc + B.c, vB);
    }
    tile = next_tile;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) my_acc += __shfl_xor_sync(FULL, my_acc, o);
  if (lane == 0 && my_acc) atomicAdd(p.acc, (unsigned long long)my_acc);
}

// Smart Monte Carlo sweep of the other chain lengths, and of even ones whose
// tiles would leave more slots empty, in the strips of strip.cuh.  2.1M
// particles of N = 33: 73.9 us a sweep in tiles, 38.5 us in strips;
// 20 cycles with 24 warps 799 us, 28 774, 32 838.
template <typename IDX>
__global__ void __launch_bounds__(896, 1) sweep_smc_strip_kernel(const SweepArgs p) {
  __shared__ uint32_t s_next;
  const int lane = threadIdx.x & 31;
  const uint32_t chunk = (p.n_items + gridDim.x - 1) / gridDim.x;
  const uint32_t item0 = blockIdx.x * chunk;
  if (threadIdx.x == 0) s_next = 0u;
  __syncthreads();
  if (idle_warp(item0, chunk, p.n_items)) return;
  chained_begin();
  const unsigned long long s64 = *p.d_sweep;
  const uint32_t sweep = (uint32_t)s64;
  uint32_t* __restrict__ nacc = ((s64 + 1ull) & 1ull) ? p.n1 : p.n0;
  const float4* __restrict__ tabA = p.smc_tab;
  const float4* __restrict__ tabB = p.smc_tab + p.g.cells;
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
    const StripPos v = nv;
    have = walk.step();
    ns = walk.place();
    strip_load(p, ns, nv);
    const bool aL = s.idx <= N_A, aR = s.idx < N_A;
    const float4* tL = aL ? tabA : tabB;
    const float4* tR = aR ? tabA : tabB;
    uint32_t w;
    const uint64_t m = (uint64_t)(s.m + (IDX)p.g.id_base);
    SmcSlot L, R;
    L.x = v.Lx; L.y = v.Ly; L.z = v.Lz;
    R.x = v.Rx; R.y = v.Ry; R.z = v.Rz;
    smc_slots(p.g, tL, tR, m - 1u, sweep, ctr3, L, R, &w);
    {  // first set: R moves against L of its own and of the next unit
      const float qx = strip_next(L.x, nv.Lx, lane), qy = strip_next(L.y, nv.Ly, lane),
                  qz = strip_next(L.z, nv.Lz, lane);
      const bool a = s.own(), b = s.next(N);
      my_acc += smc_move(p, tR, R, (a ? R.x - L.x : 0.f) + (b ? R.x - qx : 0.f),
                         (a ? R.y - L.y : 0.f) + (b ? R.y - qy : 0.f),
                         (a ? R.z - L.z : 0.f) + (b ? R.z - qz : 0.f), (float)((int)a + (int)b), s.vR);
    }
    {  // second set: L moves against R of the previous and of its own unit
      const float qx = strip_prev(R.x, bx, lane), qy = strip_prev(R.y, by, lane),
                  qz = strip_prev(R.z, bz, lane);
      const bool a = s.prev(), b = s.own();
      my_acc += smc_move(p, tL, L, (a ? L.x - qx : 0.f) + (b ? L.x - R.x : 0.f),
                         (a ? L.y - qy : 0.f) + (b ? L.y - R.y : 0.f),
                         (a ? L.z - qz : 0.f) + (b ? L.z - R.z : 0.f), (float)((int)a + (int)b), s.vL);
    }
    bx = R.x;
    by = R.y;
    bz = R.z;
    strip_store(p, s, StripPos{L.x, L.y, L.z, R.x, R.y, R.z});
    strip_count(nacc, s, L.c, R.c, aL ? 1u : 0x10000u, aR ? 1u : 0x10000u);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) my_acc += __shfl_xor_sync(FULL, my_acc, o);
  if (lane == 0 && my_acc) atomicAdd(p.acc, (unsigned long long)my_acc);
}

const void* smc_kernel_ptr(bool strip, bool big) {
  if (!strip) return (const void*)sweep_smc_pair_kernel;
  return big ? (const void*)sweep_smc_strip_kernel<uint64_t> : (const void*)sweep_smc_strip_kernel<uint32_t>;
}

}  // namespace soma
