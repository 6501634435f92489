// FP64 pair sums: density + EOS (Eq. 1), the IAD matrix, and momentum/energy
// with artificial viscosity (Eqs. 2-5).  NSUB lanes per target particle, each
// taking every NSUB-th entry of its neighbour list (entries: sph_tile.cuh) and
// gathering the neighbours' FP64 fields through L1/L2 (particles are in Morton
// cell order, so a warp's neighbours share lines); the lanes' partial sums are
// added by a fixed butterfly.  Separations are FP64 minimum-image differences
// of the positions.
//
// The FP64 pipe (2 operations per clock and SM) bounds these kernels (78-87% of
// its cycles), so FP64 operations are what is saved:
//  - S(v)^6 is evaluated on the integer pipes (sph_fixed.cuh) once per list
//    entry by the density pass, kept without its factor B_n/h^3 (Lists64::w),
//    and read back by IAD and momentum; the factor is applied per particle;
//  - the minimum image compares bit patterns as integers and adds the period
//    only in warps that hold a pair across a boundary;
//  - 1/r takes its seed from the FP32 reciprocal square root, and per-pair
//    divisions are hoisted into per-particle arrays;
//  - scalar products are block fixed point, and with S^6 (FAST) so are r^2, v
//    and 1/r, from the separation's fixed-point form;
//  - the per-target work runs on whole warps (lanes_sum).
// Per pair about 4 (density), 9 (IAD) and 26 (momentum) FP64 operations; at
// 1.07M particles 1.82, 2.86 and 7.75 ms (7.99 with C_a applied to every pair),
// where the FP64 series, products and comparisons with one thread per target took
// 7.38, 4.11 and 20.6 ms.
#include <cuda_runtime.h>
#include "sph_device.cuh"
#include "sph_fixed.cuh"
#include "sph_internal.cuh"
#include "sph_launch.cuh"
#include "sph_lanes64.cuh"
#include "sph_tile.cuh"

namespace sph {

namespace {

constexpr int kThreads64 = 128;

struct Aux64 {
  double* vol;     // m / rho
  double* X;       // P / (Omega rho^2)
  double* irq;     // alpha / (4 rho)
  double* hinv2;   // 1 / h^2
  double* mn;      // m B_n / h^3
  double* wnorm;   // B_n / h^3
  const double2* ktab;  // SPH_KERNEL_TABLE values, NULL for the exact kernel
};

struct Lists64 {
  const int32_t* nn;
  const uint32_t* nbr;
  double* w;  // h_a^3 W_ab(h_a) / B_n per entry, same layout as nbr
  int max_nb;
};

// S(v)^n at t = v^2 by the context's kernel.
__device__ __forceinline__ double shape64(double t, int n, const double2* tab) {
  if (tab) return kernel_w64_tab(t, 1.0, tab);
  return n == 6 ? fx::S6(t) : ipow(fx::S(t), n);
}

// S^6 of r^2 = R 2^k and 1 / h^2; 0 from the support's edge on (R reaches 2^60 at
// the target's own).
__device__ __forceinline__ double shape_at(int64_t R, int k, double hinv2) {
  uint64_t y;
  return (uint64_t)R >> 60 == 0 && fx::fraction_of((uint64_t)R, k, hinv2, y) ? fx::S6_at(y) : 0.0;
}

// GRADH: also the grad-h terms, Omega_a = 1 + h_a/(3 rho_a) sum_b m_b dW/dh_a.
// With dW/dh = -(3 W + v dW/dv) / h and sum_b m_b W = rho_a (self term
// included) this is Omega_a = -(2 / (3 rho_a)) sum_{b != a} m_b t dW/dt,
// t = v^2 (the self term has t = 0); X = P / (Omega rho^2) then carries it
// into Eqs. 2-3.
// FAST (the default kernel: exact, n = 6, no grad-h terms): t and S^6 in fixed
// point from the components of d, so that 4 FP64 operations per pair are left.
template <int NSUB, bool GRADH, bool FAST>
__global__ void __launch_bounds__(kThreads64) k_density64(const Grid* gp, StateView s, OutView o,
                                                          Aux64 aux, Lists64 L, int64_t n,
                                                          double Bn, int sinc_n, double gamma,
                                                          double alpha, uint32_t* err) {
  dep_enter();
  constexpr int kT = kThreads64 / NSUB;  // targets of a block
  __shared__ double sh_acc[kT], sh_g[GRADH ? kT : 1], sh_hinv2[kT];
  const Image64 im = image_of(gp);
  const int64_t a_own = blockIdx.x * (int64_t)kT + threadIdx.x;  // target finished by this thread
  const bool own = threadIdx.x < kT && a_own < n;
  const double h_own = own ? s.h[a_own] : 1.0;
  const double hinv2_own = threadIdx.x < kT ? 1.0 / (h_own * h_own) : 0.0;
  if (threadIdx.x < kT) sh_hinv2[threadIdx.x] = hinv2_own;
  const int sub = threadIdx.x % NSUB, t_loc = threadIdx.x / NSUB;
  const bool valid = blockIdx.x * (int64_t)kT + t_loc < n;
  int64_t a = valid ? blockIdx.x * (int64_t)kT + t_loc : n - 1;
  const double xa = s.x[a], ya = s.y[a], za = s.z[a];
  const int cnt = valid ? min(L.nn[a], L.max_nb) : 0;
  const uint32_t* list = L.nbr + a * L.max_nb;
  double* wrow = L.w + a * L.max_nb;
  double acc = 0.0, gsum = 0.0;
  __syncthreads();
  const double hinv2 = sh_hinv2[t_loc];
  const int ed = fx::exp_above(2.0 * s.h[a]);  // |d| < 2 h_a
  for (int k = sub; k < cnt; k += NSUB) {
    const int64_t b = entry_index(list[k]);
    double dx = s.x[b] - xa, dy = s.y[b] - ya, dz = s.z[b] - za;
    sep64(im, dx, dy, dz);
    const double mb = s.m[b];
    double w;
    if (FAST) {
      const fx::Vec3 D = vec64(dx, dy, dz, ed);
      w = shape_at(fx::dot(D, D), 2 * (ed - 1023) - 60, hinv2);
      acc += mb * w;
      wrow[k] = w;
      continue;
    }
    const double t = (dx * dx + dy * dy + dz * dz) * hinv2;
    if (GRADH) {
      double dw;
      if (sinc_n == 6)
        fx::S6_d(t, w, dw);
      else
        kernel_w64_d(t, 1.0, sinc_n, w, dw);
      gsum += mb * (t * dw);
    } else {
      w = shape64(t, sinc_n, aux.ktab);
    }
    acc += mb * w;
    wrow[k] = w;
  }
  lanes_sum<NSUB>(acc, sh_acc);
  if (GRADH) lanes_sum<NSUB>(gsum, sh_g);
  __syncthreads();
  if (!own) return;
  a = a_own;
  acc = sh_acc[threadIdx.x];
  const double norm = Bn * hinv2_own / h_own;
  const double ma = s.m[a];
  const double rho = norm * (ma + acc);  // self term: S(0) = 1
  const double p = (gamma - 1.0) * rho * s.u[a];
  const double c = sqrt(gamma * p / rho);
  o.rho[a] = rho;
  o.p[a] = p;
  o.c[a] = c;
  const double inv_rho = 1.0 / rho;
  aux.irq[a] = 0.25 * alpha * inv_rho;
  aux.vol[a] = ma * inv_rho;
  if (GRADH) {
    const double omega = -2.0 * (norm * sh_g[threadIdx.x]) * inv_rho / 3.0;
    aux.X[a] = p * inv_rho * inv_rho / omega;
    if (o.omega) o.omega[a] = omega;
  } else {
    aux.X[a] = p * inv_rho * inv_rho;
  }
  aux.hinv2[a] = hinv2_own;
  aux.mn[a] = ma * norm;
  aux.wnorm[a] = norm;
  if (!isfinite(rho) || !isfinite(c)) raise_flag(err, SPH_FLAG_NONFINITE);
}

template <int NSUB>
__global__ void __launch_bounds__(kThreads64) k_iad64(const Grid* gp, StateView s, OutView o,
                                                      Aux64 aux, Lists64 L, int64_t n, uint32_t* err) {
  dep_enter();
  constexpr int kT = kThreads64 / NSUB;  // targets of a block
  __shared__ double sums[6][kT];
  const Image64 im = image_of(gp);
  const int sub = threadIdx.x % NSUB;
  const int64_t a_pair = blockIdx.x * (int64_t)kT + threadIdx.x / NSUB;
  const bool valid = a_pair < n;
  int64_t a = valid ? a_pair : n - 1;
  const double xa = s.x[a], ya = s.y[a], za = s.z[a];
  const int cnt = valid ? min(L.nn[a], L.max_nb) : 0;
  const uint32_t* list = L.nbr + a * L.max_nb;
  const double* wrow = L.w + a * L.max_nb;
  const int ed = fx::exp_above(2.0 * s.h[a]);  // |d| < 2 h_a
  const bool mid = ed > 600 && ed < 1450;      // products stay normal
  double t00 = 0, t01 = 0, t02 = 0, t11 = 0, t12 = 0, t22 = 0;
  for (int k = sub; k < cnt; k += NSUB) {
    const int64_t b = entry_index(list[k]);
    double dx = s.x[b] - xa, dy = s.y[b] - ya, dz = s.z[b] - za;
    sep64(im, dx, dy, dz);
    // vol_b S^n d in fixed point (4 of 13 FP64 operations of a pair), in the
    // middle of the exponent range
    const double vol = aux.vol[b], sk = wrow[k];
    double wx, wy, wz;
    if (fx::middle(vol) && fx::middle(sk) && mid) {
      const fx::Mant w = fx::mant(vol) * fx::mant(sk);
      wx = fx::times(w, fx::fixed<61>(dx, ed), ed - 1023 - 61);
      wy = fx::times(w, fx::fixed<61>(dy, ed), ed - 1023 - 61);
      wz = fx::times(w, fx::fixed<61>(dz, ed), ed - 1023 - 61);
    } else {
      const double w = vol * sk;
      wx = w * dx;
      wy = w * dy;
      wz = w * dz;
    }
    t00 += wx * dx;
    t01 += wx * dy;
    t02 += wx * dz;
    t11 += wy * dy;
    t12 += wy * dz;
    t22 += wz * dz;
  }
  lanes_sum<NSUB>(t00, sums[0]);
  lanes_sum<NSUB>(t01, sums[1]);
  lanes_sum<NSUB>(t02, sums[2]);
  lanes_sum<NSUB>(t11, sums[3]);
  lanes_sum<NSUB>(t12, sums[4]);
  lanes_sum<NSUB>(t22, sums[5]);
  __syncthreads();
  a = blockIdx.x * (int64_t)kT + threadIdx.x;
  if (threadIdx.x >= kT || a >= n) return;
  const double norm = aux.wnorm[a];
  t00 = norm * sums[0][threadIdx.x];
  t01 = norm * sums[1][threadIdx.x];
  t02 = norm * sums[2][threadIdx.x];
  t11 = norm * sums[3][threadIdx.x];
  t12 = norm * sums[4][threadIdx.x];
  t22 = norm * sums[5][threadIdx.x];
  // inverse of the symmetric matrix by cofactors
  const double c00 = t11 * t22 - t12 * t12;
  const double c01 = t02 * t12 - t01 * t22;
  const double c02 = t01 * t12 - t02 * t11;
  const double c11 = t00 * t22 - t02 * t02;
  const double c12 = t01 * t02 - t00 * t12;
  const double c22 = t00 * t11 - t01 * t01;
  const double det = t00 * c00 + t01 * c01 + t02 * c02;
  double tmax = fmax(fmax(fabs(t00), fabs(t01)), fmax(fabs(t02), fabs(t11)));
  tmax = fmax(tmax, fmax(fabs(t12), fabs(t22)));
  double* out = o.iad + 6 * a;
  if (!isfinite(det) || fabs(det) <= 1e-12 * tmax * tmax * tmax) {
    raise_flag(err, SPH_FLAG_SINGULAR_IAD);
    for (int q = 0; q < 6; ++q) out[q] = 0.0;
  } else {
    const double id = 1.0 / det;
    out[0] = c00 * id;
    out[1] = c01 * id;
    out[2] = c02 * id;
    out[3] = c11 * id;
    out[4] = c12 * id;
    out[5] = c22 * id;
  }
}

// Momentum's view of a neighbour, written per launch by k_pack64: 144 bytes read
// as nine 16-byte loads where the separate arrays took 18 loads.
struct alignas(16) Rec64 {
  double x, y, z, hinv2;
  double vx, vy, vz, c;
  double m, mn;      // m, and m B_n / h^3 with the power of two of cf
  double X, irq;
  long long cf[6];   // C in block fixed point (fx::fixed), xx xy xz yy yz zz
};

__global__ void k_pack64(StateView s, OutView o, Aux64 aux, int64_t n, Rec64* rec) {
  dep_enter();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  Rec64 r;
  r.x = s.x[i];
  r.y = s.y[i];
  r.z = s.z[i];
  r.hinv2 = aux.hinv2[i];
  r.vx = s.vx[i];
  r.vy = s.vy[i];
  r.vz = s.vz[i];
  r.c = o.c[i];
  r.m = s.m[i];
  r.X = aux.X[i];
  r.irq = aux.irq[i];
  double C[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) C[q] = o.iad[6 * i + q];
  r.mn = aux.mn[i] * power_of(fix_matrix(C, r.cf));
  rec[i] = r;
}

// A lane's share of a target's pairs in plain FP64, the factors B_n/h^3 and C_a applied
// to every pair: for lanes that meet a relative velocity that is not finite or near the
// end of the exponent range, whose fixed-point products would not overflow as FP64's do.
// Its code beside the loop takes 0.5% (1.07M particles 13.52 -> 13.60 ms per step; as a
// call 13.81, after the lane sums by one thread per target 13.67).
__device__ __forceinline__ void momentum_plain(const Image64& im, const Rec64* rec,
                                               const double* iad, const Aux64& aux,
                                               const uint32_t* list, const double* wrow, int64_t a,
                                               int k0, int cnt, int step, int sinc_n, double& ax,
                                               double& ay, double& az, double& du) {
  const Rec64* ra = rec + a;
  const double* A = iad + 6 * a;
  const double wn = aux.wnorm[a];
  ax = ay = az = du = 0.0;
#pragma unroll 1
  for (int k = k0; k < cnt; k += step) {
    const int64_t b = entry_index(list[k]);
    const Rec64* rb = rec + b;
    double dx = rb->x - ra->x, dy = rb->y - ra->y, dz = rb->z - ra->z;
    sep64(im, dx, dy, dz);
    const double vx = ra->vx - rb->vx, vy = ra->vy - rb->vy, vz = ra->vz - rb->vz;
    const double r2 = dx * dx + dy * dy + dz * dz;
    const double xv = -(dx * vx + dy * vy + dz * vz);  // x_ab . v_ab
    double q = 0.0;
    if (xv < 0.0) {
      const double w = xv * rsqrt(r2);
      q = w * fma(3.0, w, -(ra->c + rb->c));
    }
    const double pa = q * ra->irq, pb = q * rb->irq;
    const double* B = iad + 6 * b;
    const double wa = rb->m * (wn * wrow[k]);
    const double wb =
        rb->m * (aux.wnorm[b] * shape64(r2 * rb->hinv2, sinc_n, aux.ktab));
    const double cax = A[0] * dx + A[1] * dy + A[2] * dz, cay = A[1] * dx + A[3] * dy + A[4] * dz,
                 caz = A[2] * dx + A[4] * dy + A[5] * dz;
    const double cbx = B[0] * dx + B[1] * dy + B[2] * dz, cby = B[1] * dx + B[3] * dy + B[4] * dz,
                 cbz = B[2] * dx + B[4] * dy + B[5] * dz;
    const double fa = wa * (ra->X + pa), fb = wb * (rb->X + pb);
    ax -= fa * cax + fb * cbx;
    ay -= fa * cay + fb * cby;
    az -= fa * caz + fb * cbz;
    du += wa * fma(0.5, pa, ra->X) * (vx * cax + vy * cay + vz * caz) +
          wb * (0.5 * pb) * (vx * cbx + vy * cby + vz * cbz);
  }
}

// Per pair, with p_a = Pi / (2 rho_a) and p_b = Pi / (2 rho_b):
//   a_a  -= m_b (W_a (X_a + p_a) C_a d + W_b (X_b + p_b) C_b d)
//   du_a += m_b (W_a (X_a + p_a / 2) v_ab.C_a d + W_b p_b / 2 v_ab.C_b d)
// The factor B_n/h_a^3 of W_a is applied to the sums, that of W_b carried by
// m_b B_n/h_b^3.  C_a d, C_b d, v.C_a d, v.C_b d and x.v (27 of the 63 FP64
// operations of a pair) are scalar products in block fixed point on the integer
// pipes, d to the power of two above 2 h_a, v to its own: their rms error, about
// 2^-60 of the largest components' product, is below FP64's.
// FAST (exact kernel, n = 6): S^6 of the neighbour's kernel, its product with
// m_b B_n/h_b^3 and x.v / r in fixed point too, except for pairs closer than
// 1/16 of the power of two above 2 h_a, which need r^2 to FP64's relative precision.
template <int NSUB, bool FAST>
__global__ void __launch_bounds__(kThreads64, 4) k_momentum64(const Grid* gp, const Rec64* rec,
                                                           StateView s, OutView o, Aux64 aux,
                                                           Lists64 L, int64_t n, int sinc_n,
                                                           uint32_t* err) {
  dep_enter();
  constexpr int kT = kThreads64 / NSUB;  // targets of a block
  __shared__ double sums[4][kT];
  const Image64 im = image_of(gp);
  const int sub = threadIdx.x % NSUB;
  const int64_t a_pair = blockIdx.x * (int64_t)kT + threadIdx.x / NSUB;
  const bool valid = a_pair < n;
  int64_t a = valid ? a_pair : n - 1;
  const Rec64* ra = rec + a;
  const double xa = ra->x, ya = ra->y, za = ra->z;
  const double vxa = ra->vx, vya = ra->vy, vza = ra->vz;
  const double Xa = ra->X, ira = ra->irq, hira = 0.5 * ira, ca = ra->c;
  const int ed = fx::exp_above(2.0 * s.h[a]);  // |d| < 2 h_a
  fx::Vec3 Ca[3];
  rows(ra->cf, Ca);
  const int cnt = valid ? min(L.nn[a], L.max_nb) : 0;
  const uint32_t* list = L.nbr + a * L.max_nb;
  const double* wrow = L.w + a * L.max_nb;
  // sum fa d and the terms of W_a, without B_n/h_a^3 (C_a is applied to the sum)
  double accx = 0, accy = 0, accz = 0, du = 0;
  double bccx = 0, bccy = 0, bccz = 0, dub = 0;     // terms of W_b
  bool far = false;  // a velocity past 2^800 or not finite
  for (int k = sub; k < cnt; k += NSUB) {
    const Rec64* rb = rec + entry_index(list[k]);
    double dx = rb->x - xa, dy = rb->y - ya, dz = rb->z - za;
    sep64(im, dx, dy, dz);
    const double vx = vxa - rb->vx, vy = vya - rb->vy, vz = vza - rb->vz;
    const fx::Vec3 D = vec64(dx, dy, dz, ed);
    const int ev = exp_max3(vx, vy, vz);
    const fx::Vec3 V = vec64(vx, vy, vz, ev);
    far |= ev > 1023 + 800;
    const int64_t vd = fx::dot(V, D);  // -x_ab . v_ab
    const int kv = ev + ed - 2 * 1023 - 60, kr = 2 * (ed - 1023) - 60;
    const int64_t R = FAST ? fx::dot(D, D) : 0;
    double wv = 0.0, wb;  // x_ab . v_ab / r where negative
    if (FAST && R >= (int64_t)1 << 52) {
      uint64_t y;
      wb = (uint64_t)R < (uint64_t)1 << 61 && fx::fraction_of((uint64_t)R, kr, rb->hinv2, y)
               ? fx::S6_at_times(y, rb->mn) : 0.0;
      if (vd > 0) wv = fx::over_root(-vd, kv, (uint64_t)R, kr);
    } else {
      const double r2 = dx * dx + dy * dy + dz * dz;
      wb = rb->mn * shape64(r2 * rb->hinv2, sinc_n, aux.ktab);
      if (vd > 0) {
        double y0, e;
        root_parts(r2, y0, e);
        const double z = fx::scaled(-vd, kv) * y0;
        wv = fma(z, e, z);
      }
    }
    double q = 0.0, pb = 0.0;
    if (vd > 0) {
      q = wv * fma(3.0, wv, -(ca + rb->c));
      pb = q * rb->irq;
    }
    const double wa = rb->m * wrow[k];
    const double fa = wa * fma(q, ira, Xa);
    const double fb = wb * (rb->X + pb);
    accx += fa * dx;
    accy += fa * dy;
    accz += fa * dz;
    {
      fx::Vec3 Uv;
#pragma unroll
      for (int i = 0; i < 3; ++i) fx::put(Uv, i, fx::dot(Ca[i], D));
      du += wa * fma(q, hira, Xa) * fx::scaled(fx::dot(V, Uv), ev - 1023);
    }
    {
      fx::Vec3 Cb[3], Uv;
      rows(rb->cf, Cb);
      int64_t U[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        U[i] = fx::dot(Cb[i], D);
        fx::put(Uv, i, U[i]);
      }
      bccx += fb * fx::scaled(U[0], 0);
      bccy += fb * fx::scaled(U[1], 0);
      bccz += fb * fx::scaled(U[2], 0);
      dub += wb * pb * fx::scaled(fx::dot(V, Uv), ev - 1023);
    }
  }
  // the powers of two of d, C_a and the products: C d = U 2^(e_C + e_d - 59),
  // v.C d = R 2^(e_v + e_C + e_d - 58)
  long long cf[6];
  const double pd = power_of(ed) * 0x1p-59;
  const double* C = o.iad + 6 * a;
  const double wn = aux.wnorm[a], pn = wn * power_of(fix_matrix(C, cf)) * pd;
  const double ax0 = accx, ay0 = accy;
  accx = fma(-wn, C[0] * ax0 + C[1] * ay0 + C[2] * accz, -pd * bccx);
  accy = fma(-wn, C[1] * ax0 + C[3] * ay0 + C[4] * accz, -pd * bccy);
  accz = fma(-wn, C[2] * ax0 + C[4] * ay0 + C[5] * accz, -pd * bccz);
  du = 2.0 * fma(pn, du, 0.5 * pd * dub);
  // past the reach of v.d (or of h) the lane's share is taken again
  if (far || ed > 1023 + 199)
    momentum_plain(im, rec, o.iad, aux, list, wrow, a, sub, cnt, NSUB, sinc_n, accx, accy, accz,
                   du);
  lanes_sum<NSUB>(accx, sums[0]);
  lanes_sum<NSUB>(accy, sums[1]);
  lanes_sum<NSUB>(accz, sums[2]);
  lanes_sum<NSUB>(du, sums[3]);
  __syncthreads();
  a = blockIdx.x * (int64_t)kT + threadIdx.x;
  if (threadIdx.x >= kT || a >= n) return;
  accx = sums[0][threadIdx.x];
  accy = sums[1][threadIdx.x];
  accz = sums[2][threadIdx.x];
  du = sums[3][threadIdx.x];
  o.ax[a] = accx;
  o.ay[a] = accy;
  o.az[a] = accz;
  o.du[a] = du;
  if (!isfinite(accx) || !isfinite(accy) || !isfinite(accz) || !isfinite(du))
    raise_flag(err, SPH_FLAG_NONFINITE);
}

inline Aux64 aux_of(sph_ctx* ctx) {
  Aux64 a;
  a.vol = ctx->vol;
  a.X = ctx->X;
  a.irq = ctx->vol + 2 * ctx->n_max;
  a.hinv2 = ctx->vol + 3 * ctx->n_max;
  a.mn = ctx->vol + 4 * ctx->n_max;
  a.wnorm = ctx->vol + 5 * ctx->n_max;
  a.ktab = ctx->prm.kernel_mode == SPH_KERNEL_TABLE ? ctx->ktab64 : nullptr;
  return a;
}

inline Lists64 lists64_of(sph_ctx* ctx) {
  Lists64 t;
  t.nn = ctx->nn;
  t.nbr = ctx->nbr;
  t.w = ctx->wcache;
  t.max_nb = ctx->prm.max_nb;
  return t;
}

// The default kernel: exact, n = 6.
inline bool fast64(const sph_ctx* ctx) {
  return ctx->prm.kernel_mode == SPH_KERNEL_EXACT && ctx->prm.sinc_n == 6.0;
}

inline unsigned blocks64(int64_t n, int nsub) {
  return (unsigned)((n * nsub + kThreads64 - 1) / kThreads64);
}

}  // namespace

void launch_density_f64(sph_ctx* ctx, const StateView& s, const OutView& o, int64_t n,
                        cudaStream_t st) {
  with_lanes64(n, [&](auto lanes) {
    constexpr int NS = decltype(lanes)::value;
    auto kern = ctx->prm.gradh ? k_density64<NS, true, false>
                               : (fast64(ctx) ? k_density64<NS, false, true>
                                              : k_density64<NS, false, false>);
    launch_dep_if(n < kEarlyPairsN, kern, blocks64(n, NS), kThreads64, 0, st, ctx->grid, s, o,
                  aux_of(ctx), lists64_of(ctx), n, ctx->Bn, (int)ctx->prm.sinc_n, ctx->prm.gamma,
                  ctx->prm.alpha, ctx->err);
  });
  ctx->launches += 1;
}

void launch_iad_f64(sph_ctx* ctx, const StateView& s, const OutView& o, int64_t n,
                    cudaStream_t st) {
  with_lanes64(n, [&](auto lanes) {
    constexpr int NS = decltype(lanes)::value;
    launch_dep_if(n < kEarlyPairsN, k_iad64<NS>, blocks64(n, NS), kThreads64, 0, st, ctx->grid, s,
                  o, aux_of(ctx), lists64_of(ctx), n, ctx->err);
  });
  ctx->launches += 1;
}

void launch_momentum_f64(sph_ctx* ctx, const StateView& s, const OutView& o, int64_t n,
                         cudaStream_t st) {
  // the records live in the hit-mask buffer of the FP32-mixed staged search
  // (a search of either form writes its own before it is read)
  static_assert(sizeof(Rec64) <= kMaskWords * sizeof(unsigned long long), "fits the mask buffer");
  Rec64* rec = reinterpret_cast<Rec64*>(ctx->masks);
  launch_dep_if(n < kEarlyPairsN, k_pack64, (unsigned)((n + 127) / 128), 128, 0, st, s, o,
                aux_of(ctx), n, rec);
  with_lanes64(n, [&](auto lanes) {
    constexpr int NS = decltype(lanes)::value;
    auto kern = fast64(ctx) ? k_momentum64<NS, true> : k_momentum64<NS, false>;
    launch_dep_if(n < kEarlyPairsN, kern, blocks64(n, NS), kThreads64, 0, st, ctx->grid, rec, s, o,
                  aux_of(ctx), lists64_of(ctx), n, (int)ctx->prm.sinc_n, ctx->err);
  });
  ctx->launches += 2;
}

}  // namespace sph
