// FP64 pair sums: density + EOS (Eq. 1), the IAD matrix, and momentum/energy
// with artificial viscosity (Eqs. 2-5).  NSUB lanes per target particle, each
// taking every NSUB-th entry of its neighbour list (entries: sph_tile.cuh) and
// gathering the neighbours' FP64 fields through L1/L2 (particles are in Morton
// cell order, so a warp's neighbours share lines); the lanes' partial sums are
// added by a fixed butterfly.  Separations are FP64 minimum-image differences
// of the positions.
//
// The FP64 pipe (2 operations per clock and SM) bounds these kernels (80-88% of
// its cycles), so FP64 operations are what is saved:
//  - S(v)^6 is evaluated on the integer pipes (sph_fixed.cuh) once per list
//    entry by the density pass, kept without its factor B_n/h^3 (Lists64::w),
//    and read back by IAD and momentum; the factor is applied per particle;
//  - the minimum image compares bit patterns as integers and adds the period
//    only in warps that hold a pair across a boundary;
//  - 1/r takes its seed from the FP32 reciprocal square root, and per-pair
//    divisions are hoisted into per-particle arrays;
//  - the per-target work runs on whole warps (lanes_sum).
// Per pair 8 (density), 13 (IAD) and 64 (momentum) FP64 operations; at 1.07M
// particles 2.64, 3.77 and 14.5 ms, where the FP64 series, FP comparisons and
// one thread per target took 7.38, 4.11 and 20.6 ms.
#include <cuda_runtime.h>
#include "sph_device.cuh"
#include "sph_fixed.cuh"
#include "sph_internal.cuh"
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

// GRADH: also the grad-h terms, Omega_a = 1 + h_a/(3 rho_a) sum_b m_b dW/dh_a.
// With dW/dh = -(3 W + v dW/dv) / h and sum_b m_b W = rho_a (self term
// included) this is Omega_a = -(2 / (3 rho_a)) sum_{b != a} m_b t dW/dt,
// t = v^2 (the self term has t = 0); X = P / (Omega rho^2) then carries it
// into Eqs. 2-3.
template <int NSUB, bool GRADH>
__global__ void __launch_bounds__(kThreads64) k_density64(const Grid* gp, StateView s, OutView o,
                                                          Aux64 aux, Lists64 L, int64_t n,
                                                          double Bn, int sinc_n, double gamma,
                                                          double alpha, uint32_t* err) {
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
  for (int k = sub; k < cnt; k += NSUB) {
    const int64_t b = entry_index(list[k]);
    double dx = s.x[b] - xa, dy = s.y[b] - ya, dz = s.z[b] - za;
    sep64(im, dx, dy, dz);
    const double t = (dx * dx + dy * dy + dz * dz) * hinv2;
    const double mb = s.m[b];
    double w;
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
  double t00 = 0, t01 = 0, t02 = 0, t11 = 0, t12 = 0, t22 = 0;
  for (int k = sub; k < cnt; k += NSUB) {
    const int64_t b = entry_index(list[k]);
    double dx = s.x[b] - xa, dy = s.y[b] - ya, dz = s.z[b] - za;
    sep64(im, dx, dy, dz);
    const double w = aux.vol[b] * wrow[k];
    const double wx = w * dx, wy = w * dy, wz = w * dz;
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

// Per pair, with p_a = Pi / (2 rho_a) and p_b = Pi / (2 rho_b):
//   a_a  -= m_b (W_a (X_a + p_a) C_a d + W_b (X_b + p_b) C_b d)
//   du_a += m_b (W_a (X_a + p_a / 2) v_ab.C_a d + W_b p_b / 2 v_ab.C_b d)
// The factor B_n/h_a^3 of W_a is applied to the sums, that of W_b carried by
// m_b B_n/h_b^3.
template <int NSUB>
__global__ void __launch_bounds__(kThreads64) k_momentum64(const Grid* gp, StateView s, OutView o,
                                                           Aux64 aux, Lists64 L, int64_t n,
                                                           int sinc_n, uint32_t* err) {
  constexpr int kT = kThreads64 / NSUB;  // targets of a block
  __shared__ double sums[4][kT];
  const Image64 im = image_of(gp);
  const int sub = threadIdx.x % NSUB;
  const int64_t a_pair = blockIdx.x * (int64_t)kT + threadIdx.x / NSUB;
  const bool valid = a_pair < n;
  int64_t a = valid ? a_pair : n - 1;
  const double xa = s.x[a], ya = s.y[a], za = s.z[a];
  const double vxa = s.vx[a], vya = s.vy[a], vza = s.vz[a];
  const double Xa = aux.X[a], ira = aux.irq[a], ca = o.c[a];
  const double* Ca = o.iad + 6 * a;
  const double a00 = Ca[0], a01 = Ca[1], a02 = Ca[2], a11 = Ca[3], a12 = Ca[4], a22 = Ca[5];
  const int cnt = valid ? min(L.nn[a], L.max_nb) : 0;
  const uint32_t* list = L.nbr + a * L.max_nb;
  const double* wrow = L.w + a * L.max_nb;
  double accx = 0, accy = 0, accz = 0, du = 0;      // terms of W_a, without B_n/h_a^3
  double bccx = 0, bccy = 0, bccz = 0, dub = 0;     // terms of W_b
  for (int k = sub; k < cnt; k += NSUB) {
    const int64_t b = entry_index(list[k]);
    double dx = s.x[b] - xa, dy = s.y[b] - ya, dz = s.z[b] - za;
    sep64(im, dx, dy, dz);
    const double r2 = dx * dx + dy * dy + dz * dz;
    const double vabx = vxa - s.vx[b], vaby = vya - s.vy[b], vabz = vza - s.vz[b];
    const double xv = -(dx * vabx + dy * vaby + dz * vabz);  // x_ab . v_ab
    double pa = 0.0, pb = 0.0;
    if (okey(xv, 0) < 0) {  // xv < 0, decided on the integer pipes
      double y0, e;
      root_parts(r2, y0, e);
      const double z = xv * y0, w = fma(z, e, z);
      const double q = w * fma(3.0, w, -(ca + o.c[b]));
      pa = q * ira;
      pb = q * aux.irq[b];
    }
    const double wa = s.m[b] * wrow[k];
    const double wb = aux.mn[b] * shape64(r2 * aux.hinv2[b], sinc_n, aux.ktab);
    // C_a d (with B_n/h_a^3) and C_b d, d = x_b - x_a
    const double Cadx = a00 * dx + a01 * dy + a02 * dz;
    const double Cady = a01 * dx + a11 * dy + a12 * dz;
    const double Cadz = a02 * dx + a12 * dy + a22 * dz;
    const double* Cb = o.iad + 6 * b;
    const double b00 = Cb[0], b01 = Cb[1], b02 = Cb[2], b11 = Cb[3], b12 = Cb[4], b22 = Cb[5];
    const double Cbdx = b00 * dx + b01 * dy + b02 * dz;
    const double Cbdy = b01 * dx + b11 * dy + b12 * dz;
    const double Cbdz = b02 * dx + b12 * dy + b22 * dz;
    const double fa = wa * (Xa + pa);
    const double fb = wb * (aux.X[b] + pb);
    accx += fa * Cadx;
    accy += fa * Cady;
    accz += fa * Cadz;
    bccx += fb * Cbdx;
    bccy += fb * Cbdy;
    bccz += fb * Cbdz;
    const double vCa = vabx * Cadx + vaby * Cady + vabz * Cadz;
    const double vCb = vabx * Cbdx + vaby * Cbdy + vabz * Cbdz;
    du += wa * fma(0.5, pa, Xa) * vCa;
    dub += wb * pb * vCb;
  }
  const double norm = aux.wnorm[a];
  lanes_sum<NSUB>(fma(-norm, accx, -bccx), sums[0]);
  lanes_sum<NSUB>(fma(-norm, accy, -bccy), sums[1]);
  lanes_sum<NSUB>(fma(-norm, accz, -bccz), sums[2]);
  lanes_sum<NSUB>(fma(norm, du, 0.5 * dub), sums[3]);
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

inline unsigned blocks64(int64_t n, int nsub) {
  return (unsigned)((n * nsub + kThreads64 - 1) / kThreads64);
}

}  // namespace

void launch_density_f64(sph_ctx* ctx, const StateView& s, const OutView& o, int64_t n,
                        cudaStream_t st) {
  with_lanes64(n, [&](auto lanes) {
    constexpr int NS = decltype(lanes)::value;
    auto kern = ctx->prm.gradh ? k_density64<NS, true> : k_density64<NS, false>;
    kern<<<blocks64(n, NS), kThreads64, 0, st>>>(
        ctx->grid, s, o, aux_of(ctx), lists64_of(ctx), n, ctx->Bn, (int)ctx->prm.sinc_n,
        ctx->prm.gamma, ctx->prm.alpha, ctx->err);
  });
  ctx->launches += 1;
}

void launch_iad_f64(sph_ctx* ctx, const StateView& s, const OutView& o, int64_t n,
                    cudaStream_t st) {
  with_lanes64(n, [&](auto lanes) {
    constexpr int NS = decltype(lanes)::value;
    k_iad64<NS><<<blocks64(n, NS), kThreads64, 0, st>>>(ctx->grid, s, o, aux_of(ctx),
                                                        lists64_of(ctx), n, ctx->err);
  });
  ctx->launches += 1;
}

void launch_momentum_f64(sph_ctx* ctx, const StateView& s, const OutView& o, int64_t n,
                         cudaStream_t st) {
  with_lanes64(n, [&](auto lanes) {
    constexpr int NS = decltype(lanes)::value;
    k_momentum64<NS><<<blocks64(n, NS), kThreads64, 0, st>>>(
        ctx->grid, s, o, aux_of(ctx), lists64_of(ctx), n, (int)ctx->prm.sinc_n, ctx->err);
  });
  ctx->launches += 1;
}

}  // namespace sph
