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
// int_0^side exp(-i s y) dy = side exp(-i s side/2) sinc(s side/2)
__device__ __forceinline__ double2 ef(double s, double side) {
  double x = 0.5 * s * side;
  double sc = fabs(x) < 1e-8 ? 1.0 - x * x / 6.0 : sin(x) / x;
  double ss, cc;
  sincos(-x, &ss, &cc);
  return make_double2(side * sc * cc, side * sc * ss);
}

struct ObsPar {
  double g1, g2;        // kappa0 x_hat1, kappa0 x_hat2
  double xh[3], e[3];   // x_hat and the polarisation vector
};

// Per direction the 1-D integrals of every mode, [C1x (nx) | S2x (nx) | S1y
// (ny) | C2y (ny)]; then each warp sums rows of E1 and E2 against them (rows
// m of E1, then of E2: nx + nx - 1), RCS_ROWS rows a block, and a last block
// per direction adds the blocks' parts in order.  (All modes of a direction in
// one block used as many SMs as there are directions: 0.12 ms for 16
// directions at 128 x 128, 0.035 ms now.)  Directions along the first axis of
// the grids, the only one that takes more than 65,535.
#define RCS_ROWS 16
__global__ void k_rcs_factors(const ObsPar* __restrict__ op, double2* __restrict__ fac, int nx,
                              int ny, double a, double b) {
  const int d = blockIdx.x, i = blockIdx.y * blockDim.x + threadIdx.x;
  if (i >= nx + ny) return;
  const bool xd = i < nx;
  const int m = xd ? i : i - nx;
  const double side = xd ? a : b, g = xd ? op[d].g1 : op[d].g2, k = m * M_PI / side;
  const double2 fm = ef(g - k, side), fp = ef(g + k, side);
  const double2 c = make_double2(0.5 * (fm.x + fp.x), 0.5 * (fm.y + fp.y));
  const double2 s = make_double2(0.5 * (fm.y - fp.y), -0.5 * (fm.x - fp.x));   // /(2i)
  double2* f = fac + (size_t)d * 2 * (nx + ny);
  if (xd) {
    f[m] = c;
    f[nx + m] = s;
  } else {
    f[2 * nx + m] = s;
    f[2 * nx + ny + m] = c;
  }
}

// grid (ndir, ceil((2 nx - 1) / RCS_ROWS)), 256 threads; part[d][block]: the
// block's parts of int E1 and int E2
__global__ void __launch_bounds__(256) k_rcs_rows(const double2* __restrict__ ap,
                                                  const double2* __restrict__ fac,
                                                  double2* __restrict__ part, int nx, int ny,
                                                  int n1, int nap) {
  __shared__ double2 red[2][8];
  const int d = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, N = ny - 1;
  const double2* E = ap + (size_t)d * nap;
  const double2* f = fac + (size_t)d * 2 * (nx + ny);
  double2 L[2] = {make_double2(0, 0), make_double2(0, 0)};
  for (int r = blockIdx.y * RCS_ROWS + warp; r < min((blockIdx.y + 1) * RCS_ROWS, 2 * nx - 1); r += 8) {
    const bool first = r < nx;
    const int m = first ? r : r - nx + 1;
    const double2* row = first ? E + (size_t)m * N - 1 : E + n1 + (size_t)(m - 1) * ny;
    const double2* fy = f + 2 * nx + (first ? 0 : ny);
    double2 s = make_double2(0, 0);
    for (int n = (first ? 1 : 0) + lane; n < ny; n += 32) s = cadd<double>(s, cmul<double>(row[n], fy[n]));
    const double2 v = cmul<double>(s, f[(first ? 0 : nx) + m]);
    L[first ? 0 : 1] = cadd<double>(L[first ? 0 : 1], v);
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    for (int off = 16; off > 0; off >>= 1) {
      L[q].x += __shfl_xor_sync(0xffffffffu, L[q].x, off);
      L[q].y += __shfl_xor_sync(0xffffffffu, L[q].y, off);
    }
    if (lane == 0) red[q][warp] = L[q];
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double2 s = make_double2(0, 0);
    for (int w = 0; w < 8; ++w) s = cadd<double>(s, red[threadIdx.x][w]);
    part[((size_t)d * gridDim.y + blockIdx.y) * 2 + threadIdx.x] = s;
  }
}

// one warp per direction
__global__ void k_rcs_final(const double2* __restrict__ part, const ObsPar* __restrict__ op,
                            double* __restrict__ sigma, int nblocks, double kappa0) {
  const int d = blockIdx.x, lane = threadIdx.x;
  double2 s1 = make_double2(0, 0), s2 = make_double2(0, 0);
  for (int k = lane; k < nblocks; k += 32) {
    s1 = cadd<double>(s1, part[((size_t)d * nblocks + k) * 2]);
    s2 = cadd<double>(s2, part[((size_t)d * nblocks + k) * 2 + 1]);
  }
  for (int off = 16; off > 0; off >>= 1) {
    s1.x += __shfl_xor_sync(0xffffffffu, s1.x, off);
    s1.y += __shfl_xor_sync(0xffffffffu, s1.y, off);
    s2.x += __shfl_xor_sync(0xffffffffu, s2.x, off);
    s2.y += __shfl_xor_sync(0xffffffffu, s2.y, off);
  }
  if (lane != 0) return;
  const ObsPar o = op[d];
  // L = (-int E2, int E1, 0)
  const double2 L[3] = {make_double2(-s2.x, -s2.y), s1, make_double2(0, 0)};
  // v = e . (x_hat x L)
  double2 v = make_double2(0, 0);
  for (int k = 0; k < 3; ++k) {
    const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
    const double2 cr = csub<double>(cscale<double>(L[k2], o.xh[k1]), cscale<double>(L[k1], o.xh[k2]));
    v = cadd<double>(v, cscale<double>(cr, o.e[k]));
  }
  sigma[d] = kappa0 * kappa0 / M_PI * cabs2<double>(v);
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
  const int nb = (2 * g.nx - 1 + RCS_ROWS - 1) / RCS_ROWS;
  const size_t b_op = al(sizeof(ObsPar) * ndir), b_sg = al(sizeof(double) * ndir);
  const size_t b_fac = al(sizeof(double2) * (size_t)ndir * 2 * (g.nx + g.ny));
  CKS(ensure_ws(ctx, &ctx->ws2, &ctx->ws2_bytes,
                b_op + b_sg + b_fac + sizeof(double2) * 2 * (size_t)ndir * nb));
  char* w = (char*)ctx->ws2;
  ObsPar* op = (ObsPar*)w;
  double* sg = (double*)(w + b_op);
  double2* fac = (double2*)(w + b_op + b_sg);
  double2* part = (double2*)(w + b_op + b_sg + b_fac);
  CK(cudaMemcpyAsync(op, hp.data(), sizeof(ObsPar) * ndir, cudaMemcpyHostToDevice, ctx->stream));
  {
    KScope ks_(ctx, KC_RHS);
    k_rcs_factors<<<dim3(ndir, (g.nx + g.ny + 127) / 128), 128, 0, ctx->stream>>>(op, fac, g.nx, g.ny,
                                                                               g.a, g.b);
  }
  {
    KScope ks_(ctx, KC_RHS);
    k_rcs_rows<<<dim3(ndir, nb), 256, 0, ctx->stream>>>(ap, fac, part, g.nx, g.ny, g.n1, g.nap);
  }
  {
    KScope ks_(ctx, KC_RHS);
    k_rcs_final<<<ndir, 32, 0, ctx->stream>>>(part, op, sg, nb, ctx->kappa0);
  }
  CK(cudaGetLastError());
  CK(cudaMemcpyAsync(sigma, sg, sizeof(double) * ndir, cudaMemcpyDeviceToHost, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  return CAVITY_OK;
}
