// Right-hand side of (EJ1)/(uT1) (row 2 of the design table, "forward
// transform of the excitation") and the backscatter RCS.
//
// RHS: g1 = (h/q) 2i(alpha1 p3 + beta p1) g~1, g2 = (h/c) 2i(alpha2 p3 + beta p2) g~2
// (c1mn and Appendix A), where g~ are the Galerkin tests (nosig) of the plane
// wave exp(i(alpha1 x1 + alpha2 x2)) taken with the trapezoid rule on the
// aperture nodes.  The test integral is separable, so per direction four 1-D
// sums  sum_p w_p {cos,sin}(m pi p/Nx) exp(i alpha1 x1_p)  (and the x2
// counterparts) are formed and multiplied out.
//
// RCS: L = int_Gamma (z x E) exp(-i kappa0 x_hat . y) dy with the exact 1-D
// integrals of cos/sin(m pi y/a) exp(-i g y), then
// sigma = (kappa0^2/pi) |e . (x_hat x L)|^2 (derived from (EGa2)).
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"

struct DirPar {
  double a1, a2, A1r, A1i, A2r, A2i;  // alpha1, alpha2, 2i(alpha1 p3 + beta p1), 2i(...)
};

// incident wave of Sec. 7: d = -(sin t cos f, sin t sin f, cos t), q = kappa0 d,
// p = cos(alpha) theta_hat + sin(alpha) phi_hat
static DirPar dir_params(double kappa0, double t, double f, double al) {
  double st = std::sin(t), ct = std::cos(t), sf = std::sin(f), cf = std::cos(f);
  double a1 = -kappa0 * st * cf, a2 = -kappa0 * st * sf, beta = kappa0 * ct;
  double th[3] = {ct * cf, ct * sf, -st}, ph[3] = {-sf, cf, 0.0};
  double p[3];
  for (int k = 0; k < 3; ++k) p[k] = std::cos(al) * th[k] + std::sin(al) * ph[k];
  DirPar d;
  d.a1 = a1;
  d.a2 = a2;
  double s1 = a1 * p[2] + beta * p[0], s2 = a2 * p[2] + beta * p[1];
  d.A1r = 0.0; d.A1i = 2.0 * s1;
  d.A2r = 0.0; d.A2i = 2.0 * s2;
  return d;
}

// fac layout per direction: [cx (nx) | sx (nx) | cy (ny+1) | sy (ny+1)]
// cx[m] = sum_p w_p cos(m pi p/nx) e^{i a1 x_p}, m = 0..nx-1;  sx[m] likewise
// with sin (index m, m = 1..nx-1 used); cy, sy over n = 0..ny.
// With cos = (e^{+} + e^{-})/2 both reduce to the trapezoid sum of a geometric
// progression, in closed form:
//   T(th) = 1/2 + z + ... + z^{N-1} + z^N/2 = (i/2) cot(th/2) (1 - z^N),  z = e^{i th},
//   th = (alpha side +- pi m)/N,  z^N = (-1)^m e^{i alpha side};
// where |sin(th/2)| < 1e-3, 1 - z^N is formed from N th instead (2 sin^2 and
// sin do not cancel; a term-by-term sum there kept whole warps waiting for one
// lane: 0.24 ms for 16 directions at 128 x 128, 0.011 ms now).
__device__ double2 trap_progression(double th, int N, double2 zN) {
  double s, c;
  sincos(0.5 * th, &s, &c);
  if (fabs(s) < 1e-3) {
    if (s == 0.0) return make_double2((double)N, 0.0);
    double hs, hc;
    sincos(0.5 * N * th, &hs, &hc);   // 1 - cos x = 2 sin^2(x/2), sin x = 2 sin cos
    const double ct = c / s;
    return make_double2(ct * hs * hc, ct * hs * hs);
  }
  const double ct = 0.5 * c / s;
  return make_double2(ct * zN.y, ct * (1.0 - zN.x));
}

__global__ void k_rhs_factors(const DirPar* __restrict__ dp, double2* __restrict__ fac, int nx,
                              int ny, double a, double b) {
  const int d = blockIdx.y, which = blockIdx.z;
  const int per = 2 * nx + 2 * (ny + 1);
  const bool xdir = which < 2;
  const int nint = xdir ? nx : ny;
  const int count = xdir ? nx : ny + 1;
  const double side = xdir ? a : b;
  const double al = xdir ? dp[d].a1 : dp[d].a2;
  const bool isc = (which == 0 || which == 2);
  const int off = which == 0 ? 0 : which == 1 ? nx : which == 2 ? 2 * nx : 2 * nx + ny + 1;
  double es, ec;
  sincos(al * side, &es, &ec);
  const double w = side / nint;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < count; m += gridDim.x * blockDim.x) {
    const double sg = (m & 1) ? -1.0 : 1.0;
    const double2 zN = make_double2(sg * ec, sg * es);
    const double2 gp = trap_progression((al * side + M_PI * m) / nint, nint, zN);
    const double2 gm = trap_progression((al * side - M_PI * m) / nint, nint, zN);
    double2 r;
    if (isc) r = make_double2(0.5 * w * (gp.x + gm.x), 0.5 * w * (gp.y + gm.y));
    else r = make_double2(0.5 * w * (gp.y - gm.y), -0.5 * w * (gp.x - gm.x));
    fac[(size_t)d * per + off + m] = r;
  }
}

__global__ void k_rhs_assemble(const DirPar* __restrict__ dp, const double2* __restrict__ fac,
                               double2* __restrict__ out, int nx, int ny, int n1, int n2, int nap,
                               int ndir, double a, double b, double h) {
  long long gid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (gid >= (long long)ndir * nap) return;
  const int d = (int)(gid / nap), i = (int)(gid - (long long)d * nap);
  const int N = ny - 1;
  const int per = 2 * nx + 2 * (ny + 1);
  const double2* f = fac + (size_t)d * per;
  const double2* cx = f;
  const double2* sx = f + nx;
  const double2* cy = f + 2 * nx;
  const double2* sy = f + 2 * nx + ny + 1;
  const double ab = a * b;
  double2 r = make_double2(0, 0);
  if (i < n1) {
    int m = i / N, n = i - m * N + 1;
    double2 g = cmul<double>(cx[m], sy[n]);
    double s = h / (m == 0 ? ab / 2 : ab / 4);
    r = cscale<double>(cmul<double>(make_double2(dp[d].A1r, dp[d].A1i), g), s);
  } else if (i < n1 + n2) {
    int ii = i - n1;
    int m = ii / (N + 1) + 1, n = ii - (m - 1) * (N + 1);
    double2 g = cmul<double>(sx[m], cy[n]);
    double s = h / (n == 0 ? ab / 2 : ab / 4);
    r = cscale<double>(cmul<double>(make_double2(dp[d].A2r, dp[d].A2i), g), s);
  }
  out[gid] = r;
}

cavity_status launch_rhs(cavity_ctx* ctx, int ndir, const double* theta, const double* phi,
                         const double* alpha, double2* out) {
  const Geo& g = ctx->g;
  std::vector<DirPar> hp(ndir);
  for (int d = 0; d < ndir; ++d) hp[d] = dir_params(ctx->kappa0, theta[d], phi[d], alpha[d]);
  const int per = 2 * g.nx + 2 * (g.ny + 1);
  size_t need = sizeof(DirPar) * ndir + sizeof(double2) * (size_t)per * ndir + 256;
  CKS(ensure_ws(ctx, &ctx->ws2, &ctx->ws2_bytes, need));
  DirPar* dp = (DirPar*)ctx->ws2;
  double2* fac = (double2*)((char*)ctx->ws2 + ((sizeof(DirPar) * ndir + 255) / 256) * 256);
  CK(cudaMemcpyAsync(dp, hp.data(), sizeof(DirPar) * ndir, cudaMemcpyHostToDevice, ctx->stream));
  int bx = (std::max(g.nx, g.ny + 1) + 127) / 128;
  {
    KScope ks_(ctx, KC_RHS);
    k_rhs_factors<<<dim3(bx, ndir, 4), 128, 0, ctx->stream>>>(dp, fac, g.nx, g.ny, g.a, g.b);
  }
  long long tot = (long long)ndir * g.nap;
  {
    KScope ks_(ctx, KC_RHS);
    k_rhs_assemble<<<(unsigned)((tot + 255) / 256), 256, 0, ctx->stream>>>(
        dp, fac, out, g.nx, g.ny, g.n1, g.n2, g.nap, ndir, g.a, g.b, g.h);
  }
  CK(cudaGetLastError());
  // the host parameter array must outlive the copy
  CK(cudaStreamSynchronize(ctx->stream));
  return CAVITY_OK;
}

// ------------------------------------------------------------------ RCS
// (Sums and products whose fusing the compiler could choose by the kernel they are
// inlined into are written as such: two kernels below share them to the last bit.)
// int_0^side exp(-i s y) dy = side exp(-i s side/2) sinc(s side/2)
__device__ __forceinline__ double2 ef(double s, double side) {
  const double x = 0.5 * s * side;
  double sn, cs;
  sincos(x, &sn, &cs);
  const double sc = fabs(x) < 1e-8 ? 1.0 - x * x / 6.0 : sn / x;
  return make_double2(__dmul_rn(side * sc, cs), __dmul_rn(-side * sc, sn));
}

struct ObsPar {
  double g1, g2;        // kappa0 x_hat1, kappa0 x_hat2
  double xh[3], e[3];   // x_hat and the polarisation vector
};

// Per direction the 1-D integrals of every mode, [C1x (nx) | S2x (nx) | S1y
// (ny) | C2y (ny)], against which the rows of E1 and of E2 are summed by blocks
// of 256 threads in units of RCS_PASSES passes (32 lanes a row, or as many as a
// short row has entries).  A thread adds its parts of the units in order, then
// the threads are added: once per direction, since with two FP64 lanes per SM
// that takes as long as 20 terms of the sum.
//
// Two ways, with the same operations in the same order, which depends on the
// grid alone (a direction's result has the same bits in any batch): one block a
// direction for all of it (k_rcs_whole), where there are directions for two
// blocks on every SM or little to do; else the units of a direction on blocks of
// their own, which store every thread's part (k_rcs_factors, k_rcs_units,
// k_rcs_final: two launches and that traffic more, but as many SMs as there are
// units).
// Directions go along the first axis of the grids, the only one that takes more
// than 65,535.  Measured on a GB300, a call's us with every unit's sum reduced in
// its block, and now: 64 x 64, 300 directions 142 -> 99; 256 x 256, 64 237 -> 139;
// 1024 x 4, 300 988 -> 156; 64 x 64, one 48 -> 48; 1024 x 1024, one 83 -> 87.  One
// block a direction against its units on many: 64 x 64, one direction 68 and 48,
// 300 99 and 126; 16 x 16, one 41 and 52.
#define RCS_PASSES 2
struct RcsUnits {
  int lpr, rows, n1, n2;   // lanes per row, rows per unit, units of E1 (nx rows) and of E2 (nx - 1)
  RcsUnits(int nx, int ny) {
    lpr = ny < 32 ? ny : 32;
    rows = RCS_PASSES * (256 / lpr);
    n1 = (nx + rows - 1) / rows;
    n2 = (nx - 1 + rows - 1) / rows;
  }
};

// integrals of mode i of [x modes | y modes] into f
__device__ __forceinline__ void rcs_mode(int i, const ObsPar& o, double2* f, int nx, int ny, double a,
                                         double b) {
  const bool xd = i < nx;
  const int m = xd ? i : i - nx;
  const double side = xd ? a : b, g = xd ? o.g1 : o.g2, k = m * M_PI / side;
  const double2 fm = ef(g - k, side), fp = ef(g + k, side);
  const double2 c = make_double2(0.5 * __dadd_rn(fm.x, fp.x), 0.5 * __dadd_rn(fm.y, fp.y));
  const double2 s = make_double2(0.5 * __dsub_rn(fm.y, fp.y), -0.5 * __dsub_rn(fm.x, fp.x));   // /(2i)
  if (xd) {
    f[m] = c;
    f[nx + m] = s;
  } else {
    f[2 * nx + m] = s;
    f[2 * nx + ny + m] = c;
  }
}

// s + a b, four multiply-adds
__device__ __forceinline__ double2 rcs_fma(double2 a, double2 b, double2 s) {
  return make_double2(__fma_rn(a.x, b.x, __fma_rn(-a.y, b.y, s.x)),
                      __fma_rn(a.x, b.y, __fma_rn(a.y, b.x, s.y)));
}
__device__ __forceinline__ double2 rcs_add(double2 a, double2 b) {
  return make_double2(__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y));
}

// thread t's part of unit u of E1 (FIRST) or E2
template <bool FIRST>
__device__ __forceinline__ double2 rcs_unit(int u, int t, const double2* __restrict__ E,
                                            const double2* f, int nx, int ny, int n1,
                                            const RcsUnits& un) {
  const int lr = 31 - __clz(un.lpr);   // a power of two
  const int sub = t >> lr, lane = t & (un.lpr - 1);
  const double2* fy = f + 2 * nx + (FIRST ? 0 : ny);
  double2 acc = make_double2(0, 0);
#pragma unroll
  for (int k = 0; k < RCS_PASSES; ++k) {
    const int m = u * un.rows + k * (256 >> lr) + sub + (FIRST ? 0 : 1);
    if (m >= nx) break;
    const double2* row = FIRST ? E + (size_t)m * (ny - 1) - 1 : E + n1 + (size_t)(m - 1) * ny;
    double2 s = make_double2(0, 0);
#pragma unroll 4
    for (int n = (FIRST ? 1 : 0) + lane; n < ny; n += un.lpr) s = rcs_fma(row[n], fy[n], s);
    acc = rcs_fma(s, f[(FIRST ? 0 : nx) + m], acc);
  }
  return acc;
}

// cross-section from int E1 and int E2
__device__ __noinline__ double rcs_sigma(double2 s1, double2 s2, const ObsPar* __restrict__ op,
                                         double kappa0) {
  const ObsPar o = *op;
  // L = (-int E2, int E1, 0)
  const double2 L[3] = {make_double2(-s2.x, -s2.y), s1, make_double2(0, 0)};
  // v = e . (x_hat x L)
  double2 v = make_double2(0, 0);
  for (int k = 0; k < 3; ++k) {
    const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
    const double2 cr = csub<double>(cscale<double>(L[k2], o.xh[k1]), cscale<double>(L[k1], o.xh[k2]));
    v = cadd<double>(v, cscale<double>(cr, o.e[k]));
  }
  return kappa0 * kappa0 / M_PI * cabs2<double>(v);
}
// the 256 threads' int E1 (a) and int E2 (b) into direction d's cross-section
__device__ __forceinline__ void rcs_finish(double2 a, double2 b, const ObsPar* __restrict__ op, int d,
                                           double* __restrict__ sigma, double kappa0) {
  __shared__ double2 red[2][8];
  for (int off = 16; off > 0; off >>= 1) {
    a.x += __shfl_xor_sync(0xffffffffu, a.x, off);
    a.y += __shfl_xor_sync(0xffffffffu, a.y, off);
    b.x += __shfl_xor_sync(0xffffffffu, b.x, off);
    b.y += __shfl_xor_sync(0xffffffffu, b.y, off);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = a;
    red[1][threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  double2 s1 = red[0][0], s2 = red[1][0];
  for (int k = 1; k < 8; ++k) {
    s1 = rcs_add(s1, red[0][k]);
    s2 = rcs_add(s2, red[1][k]);
  }
  sigma[d] = rcs_sigma(s1, s2, op + d, kappa0);
}

// grid ndir, 256 threads, 2 (nx + ny) complex values of shared memory
__global__ void __launch_bounds__(256) k_rcs_whole(const double2* __restrict__ ap,
                                                   const ObsPar* __restrict__ op,
                                                   double* __restrict__ sigma, int nx, int ny,
                                                   int n1, int nap, double a, double b,
                                                   RcsUnits un, double kappa0) {
  extern __shared__ double2 sm_f[];
  const int d = blockIdx.x, t = threadIdx.x;
  for (int i = t; i < nx + ny; i += 256) rcs_mode(i, op[d], sm_f, nx, ny, a, b);
  __syncthreads();
  const double2* E = ap + (size_t)d * nap;
  double2 s1 = make_double2(0, 0), s2 = make_double2(0, 0);
  for (int u = 0; u < un.n1; ++u) s1 = rcs_add(s1, rcs_unit<true>(u, t, E, sm_f, nx, ny, n1, un));
  for (int u = 0; u < un.n2; ++u) s2 = rcs_add(s2, rcs_unit<false>(u, t, E, sm_f, nx, ny, n1, un));
  rcs_finish(s1, s2, op, d, sigma, kappa0);
}

// grid (ndir, ceil((nx + ny) / 128))
__global__ void k_rcs_factors(const ObsPar* __restrict__ op, double2* __restrict__ fac, int nx,
                              int ny, double a, double b) {
  const int d = blockIdx.x, i = blockIdx.y * blockDim.x + threadIdx.x;
  if (i < nx + ny) rcs_mode(i, op[d], fac + (size_t)d * 2 * (nx + ny), nx, ny, a, b);
}
// grid (ndir, units), 256 threads; part[d][unit][thread]
__global__ void __launch_bounds__(256) k_rcs_units(const double2* __restrict__ ap,
                                                   const double2* __restrict__ fac,
                                                   double2* __restrict__ part, int nx, int ny,
                                                   int n1, int nap, RcsUnits un) {
  const int d = blockIdx.x, u = blockIdx.y, t = threadIdx.x;
  const double2* E = ap + (size_t)d * nap;
  const double2* f = fac + (size_t)d * 2 * (nx + ny);
  part[((size_t)d * gridDim.y + u) * 256 + t] =
      u < un.n1 ? rcs_unit<true>(u, t, E, f, nx, ny, n1, un)
                : rcs_unit<false>(u - un.n1, t, E, f, nx, ny, n1, un);
}
// grid ndir, 256 threads
__global__ void __launch_bounds__(256) k_rcs_final(const double2* __restrict__ part,
                                                   const ObsPar* __restrict__ op,
                                                   double* __restrict__ sigma, RcsUnits un,
                                                   double kappa0) {
  const int d = blockIdx.x;
  const double2* p = part + (size_t)d * (un.n1 + un.n2) * 256 + threadIdx.x;
  double2 s1 = make_double2(0, 0), s2 = make_double2(0, 0);
#pragma unroll 8
  for (int u = 0; u < un.n1; ++u) s1 = rcs_add(s1, p[(size_t)u * 256]);
  p += (size_t)un.n1 * 256;
#pragma unroll 8
  for (int u = 0; u < un.n2; ++u) s2 = rcs_add(s2, p[(size_t)u * 256]);
  rcs_finish(s1, s2, op, d, sigma, kappa0);
}

// whether one block takes a direction
static bool rcs_whole(int ndir, int nx, int ny) {
  return ndir >= 2 * sm_count() || nx * ny <= 512;
}

cavity_status launch_rcs(cavity_ctx* ctx, int ndir, const double2* ap, const double* th,
                         const double* ph, int pol, double* sigma) {
  const Geo& g = ctx->g;
  std::vector<ObsPar> hp(ndir);
  for (int d = 0; d < ndir; ++d) {
    double st = std::sin(th[d]), ct = std::cos(th[d]), sf = std::sin(ph[d]), cf = std::cos(ph[d]);
    ObsPar& o = hp[d];
    o.xh[0] = st * cf; o.xh[1] = st * sf; o.xh[2] = ct;
    o.g1 = ctx->kappa0 * o.xh[0];
    o.g2 = ctx->kappa0 * o.xh[1];
    if (pol == CAVITY_POL_THETA) { o.e[0] = ct * cf; o.e[1] = ct * sf; o.e[2] = -st; }
    else { o.e[0] = -sf; o.e[1] = cf; o.e[2] = 0.0; }
  }
  auto al = [](size_t v) { return (v + 255) / 256 * 256; };
  const RcsUnits un(g.nx, g.ny);
  const bool whole = rcs_whole(ndir, g.nx, g.ny);
  const size_t b_op = al(sizeof(ObsPar) * ndir), b_sg = al(sizeof(double) * ndir);
  const size_t b_fac = whole ? 0 : al(sizeof(double2) * (size_t)ndir * 2 * (g.nx + g.ny));
  const size_t b_part = whole ? 0 : sizeof(double2) * 256 * (size_t)ndir * (un.n1 + un.n2);
  CKS(ensure_ws(ctx, &ctx->ws2, &ctx->ws2_bytes, b_op + b_sg + b_fac + b_part));
  char* w = (char*)ctx->ws2;
  ObsPar* op = (ObsPar*)w;
  double* sg = (double*)(w + b_op);
  double2* fac = (double2*)(w + b_op + b_sg);
  double2* part = (double2*)(w + b_op + b_sg + b_fac);
  CK(cudaMemcpyAsync(op, hp.data(), sizeof(ObsPar) * ndir, cudaMemcpyHostToDevice, ctx->stream));
  if (whole) {
    static DeviceFlag done;
    if (!done) {
      CK(allow_max_smem(k_rcs_whole));
      done.set();
    }
    KScope ks_(ctx, KC_RHS);
    k_rcs_whole<<<ndir, 256, sizeof(double2) * 2 * (g.nx + g.ny), ctx->stream>>>(
        ap, op, sg, g.nx, g.ny, g.n1, g.nap, g.a, g.b, un, ctx->kappa0);
  } else {
    {
      KScope ks_(ctx, KC_RHS);
      k_rcs_factors<<<dim3(ndir, (g.nx + g.ny + 127) / 128), 128, 0, ctx->stream>>>(
          op, fac, g.nx, g.ny, g.a, g.b);
    }
    {
      KScope ks_(ctx, KC_RHS);
      k_rcs_units<<<dim3(ndir, un.n1 + un.n2), 256, 0, ctx->stream>>>(ap, fac, part, g.nx, g.ny,
                                                                      g.n1, g.nap, un);
    }
    {
      KScope ks_(ctx, KC_RHS);
      k_rcs_final<<<ndir, 256, 0, ctx->stream>>>(part, op, sg, un, ctx->kappa0);
    }
  }
  CK(cudaGetLastError());
  CK(cudaMemcpyAsync(sigma, sg, sizeof(double) * ndir, cudaMemcpyDeviceToHost, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  return CAVITY_OK;
}
