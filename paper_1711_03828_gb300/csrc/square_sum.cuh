// square_sum.cuh -- sums of squared distances between particles, as exact as
// FP64 additions or more so, without the FP64 pipe (internal).
#pragma once

#include "common.cuh"

namespace soma {

// Sum of |r - s|^2 over pairs of FP32 positions.  A component's difference is
// d + err exactly (the two-sum of Knuth, The Art of Computer Programming 2,
// 4.2.2; err is 0 unless the positions lie near the origin of the axis).  Where
// both parts are multiples of 2^-26 and the difference is below 32 in
// magnitude (positions of |x| >= 1/8 are such multiples) it is squared as a
// 32-bit integer, and the sum is kept in units of 2^-52 in two 64-bit words (the
// low and high halves of every term apart, so that 2^31 terms fit).  A pair with
// another component is added in FP64, as all of them were before; a warp pays
// for that whole, so it has to be rare: with every pair of err != 0 there, which
// the ends of chains near the origin often are, chain_obs_kernel took 140 us for
// 16.8M particles.
struct SquareSum {
  unsigned long long lo = 0, hi = 0;
  double rest = 0.0;

  __device__ __forceinline__ static bool exact(float a, float b, int& i) {
    const float s = __fsub_rn(a, b), c = __fsub_rn(s, a);
    const float err = __fsub_rn(__fsub_rn(a, __fsub_rn(s, c)), __fadd_rn(b, c));
    const float t = __fmul_rn(s, 67108864.f);   // 2^26, exact
    i = __float2int_rn(t);
    bool ok = fabsf(s) < 31.f && __int2float_rn(i) == t;
    if (err != 0.f) {
      const float e = __fmul_rn(err, 67108864.f);   // |err| <= ulp(s)/2: far below 2^31
      const int j = __float2int_rn(e);
      ok = ok && __int2float_rn(j) == e;
      i += j;
    }
    return ok;
  }

  __device__ __forceinline__ void add(float ax, float ay, float az, float bx, float by, float bz) {
    int ix, iy, iz;
    const bool ok = exact(ax, bx, ix) & exact(ay, by, iy) & exact(az, bz, iz);
    if (ok) {
      const unsigned long long u = (unsigned long long)((long long)ix * ix) +
                                   (unsigned long long)((long long)iy * iy) +
                                   (unsigned long long)((long long)iz * iz);   // < 3 2^62
      lo += (uint32_t)u;
      hi += u >> 32;
    } else {
      const double dx = (double)ax - (double)bx, dy = (double)ay - (double)by,
                   dz = (double)az - (double)bz;
      rest += dx * dx + dy * dy + dz * dz;
    }
  }

  __device__ __forceinline__ double value() const {
    // (hi 2^32 + lo) 2^-52
    return fma((double)hi, 9.5367431640625e-07, (double)lo * 2.220446049250313e-16) + rest;
  }
};

// FP64 block reduction in a fixed order (deterministic for a fixed launch).
template <int K>
__device__ __forceinline__ void block_sum(double (&v)[K], double* sh /* K*32 */) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k)
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(FULL, v[k], o);
  if (lane == 0)
    for (int k = 0; k < K; ++k) sh[k * 32 + wid] = v[k];
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    for (int k = 0; k < K; ++k) {
      double t = lane < nw ? sh[k * 32 + lane] : 0.0;
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(FULL, t, o);
      v[k] = t;
    }
  }
}

}  // namespace soma
