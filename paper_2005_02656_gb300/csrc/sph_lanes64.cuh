// What the FP64 pair kernels (sph_pairs_fp64.cu) and their reverse kernels
// (sph_adjoint.cu) share: the minimum image decided on the integer pipes,
// vectors and matrices in block fixed point, and the split of a target's
// neighbours over lanes.
#pragma once

#include <type_traits>

#include "sph_device.cuh"
#include "sph_fixed.cuh"
#include "sph_internal.cuh"

namespace sph {

// Periods of the minimum image: L per axis and the bit pattern of L / 2
// (all ones on open axes, which no |d| exceeds).
struct Image64 {
  double L[3];
  unsigned long long half[3];
};

__device__ __forceinline__ Image64 image_of(const Grid* g) {
  Image64 im;
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    im.L[ax] = g->Lbox[ax];
    im.half[ax] = g->periodic[ax] ? (unsigned long long)__double_as_longlong(g->halfL[ax]) : ~0ull;
  }
  return im;
}

__device__ __forceinline__ bool beyond(double d, unsigned long long half) {
  return ((unsigned long long)__double_as_longlong(d) & 0x7fffffffffffffffull) > half;
}

// FP64 minimum-image separation x_b - x_a: min_image's subtraction or addition
// of the period where |d| > L/2, the test on the bit patterns of |d| and L/2
// (ordered as the values are).  The FP64 additions sit behind a warp vote, so
// that the warps away from the periodic boundaries skip them.
__device__ __forceinline__ void sep64(const Image64& im, double& dx, double& dy, double& dz) {
  const bool fx = beyond(dx, im.half[0]), fy = beyond(dy, im.half[1]), fz = beyond(dz, im.half[2]);
  if (__any_sync(__activemask(), fx | fy | fz)) {
    if (fx) dx += __double2hiint(dx) < 0 ? im.L[0] : -im.L[0];
    if (fy) dy += __double2hiint(dy) < 0 ? im.L[1] : -im.L[1];
    if (fz) dz += __double2hiint(dz) < 0 ? im.L[2] : -im.L[2];
  }
}

// Power of two above three components (fx::exp_above; over 2047: not finite).
__device__ __forceinline__ int exp_max3(double x, double y, double z) {
  return max(fx::exp_above(x), max(fx::exp_above(y), fx::exp_above(z)));
}

// The same, or fx::kNotFinite.
__device__ __forceinline__ int exp_above3(double x, double y, double z) {
  const int e = exp_max3(x, y, z);
  return e <= 2047 ? e : fx::kNotFinite;
}

// A vector in block fixed point with the given power of two.
__device__ __forceinline__ fx::Vec3 vec64(double x, double y, double z, int eb) {
  fx::Vec3 v;
  fx::put(v, 0, fx::fixed<61>(x, eb));
  fx::put(v, 1, fx::fixed<61>(y, eb));
  fx::put(v, 2, fx::fixed<61>(z, eb));
  return v;
}

// C (6 entries) as block fixed point; the exponent field of the power of two
// above its largest entry, or fx::kNotFinite (and zero entries).
__device__ __forceinline__ int fix_matrix(const double* C, long long cf[6]) {
  int eb = 1;
#pragma unroll
  for (int q = 0; q < 6; ++q) eb = max(eb, fx::exp_above(C[q]));
  if (eb > 2047) eb = fx::kNotFinite;
#pragma unroll
  for (int q = 0; q < 6; ++q) cf[q] = fx::fixed<60>(C[q], eb);
  return eb;
}

// 2^(eb - 1023) for eb of fix_matrix (not finite: NaN).
__device__ __forceinline__ double power_of(int eb) {
  if (eb == fx::kNotFinite) return __longlong_as_double(0x7ff8000000000000LL);
  return eb < 2047 ? __hiloint2double(eb << 20, 0) : 2.0 * __hiloint2double(2046 << 20, 0);
}

// Rows of a symmetric matrix in block fixed point.
__device__ __forceinline__ void rows(const long long cf[6], fx::Vec3 R[3]) {
  constexpr int at[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) fx::put(R[i], j, cf[at[i][j]]);
}

// Sum over the NSUB lanes of a target, left in sums[target of the block].
// The per-target work around the pair loop (divisions, the matrix inverse: as
// many FP64 instructions as a few pairs) then runs on whole warps, one thread
// per target, instead of one lane in NSUB.
template <int NSUB>
__device__ __forceinline__ void lanes_sum(double v, double* sums) {
#pragma unroll
  for (int o = NSUB / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (threadIdx.x % NSUB == 0) sums[threadIdx.x / NSUB] = v;
}

// Lanes per target.  More lanes keep the FP64 pipes of all SMs busy at small n
// and cost lane sums and part-filled last turns of the lists at large n.
// Density + IAD + momentum with 4 / 8 / 16 lanes (us): 1,728 particles 167 / 103 /
// 71, 4,096: 168 / 114 / 97, 8,000: 186 / 152 / 154, 13,824: 219 / 232 / 235,
// 21,952: 357 / 338 / 337, 64,000: 800 / 803 / 884, 1.07M: 12,350 / 13,130 / -.
// (At 13,824 four lanes are ahead: momentum's 432 blocks are one wave of up to 608,
// with eight and sixteen lanes 1.4 and 2.8 waves, which no line in n follows; the first
// line parts sixteen lanes from eight, level from 8,000 to 21,952 and 15% apart at 4,096.
// At 32,768 four lanes take 451 against 457 us by themselves, but the step between host
// copies 736 against 699.)  20 steps and their gradient (ms): 21.8 / 16.5 / 16.6 at 4,096,
// 69.1 / 63.4 / 67.6 at 32,768, 180.5 / 181.6 / 203 at 110,592.
inline int lanes64(int64_t n) { return n < 16384 ? 16 : n < 131072 ? 8 : 4; }

// f(integral_constant<int, lanes>) for n particles.
template <class F>
inline void with_lanes64(int64_t n, F f) {
  switch (lanes64(n)) {
    case 4: f(std::integral_constant<int, 4>()); break;
    case 8: f(std::integral_constant<int, 8>()); break;
    default: f(std::integral_constant<int, 16>());
  }
}

}  // namespace sph
