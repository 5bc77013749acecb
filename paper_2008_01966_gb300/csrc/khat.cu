// Kernel table of Sec. 5.2: the 2-D Fourier transform of the truncated
// free-space Green's function,
//     F(G)(rho) = 1/2 int_0^R J0(2 pi rho r) exp(i kappa0 r) dr,
// R = sqrt(2) max(a, b), at rho = |(j1/Lx, j2/Ly)| for the quarter box
// 0 <= j1 < Px/2, 0 <= j2 < Py/2 (the table is even in j1 and in j2).
// (The paper prints 1/(4 pi) in front of the radial integral; the angular
// integral contributes 2 pi J0, hence the 1/2.)
//
// The integrand is entire, so composite Gauss-Legendre quadrature converges
// geometrically: panels no wider than pi / (2 pi rho + |kappa0|), 16 nodes
// each.  One warp per table entry, lanes striding over panels, a fixed-order
// shuffle reduction (deterministic).  FP64 throughout.  Entries of large
// argument away from the ridge 2 pi rho = kappa0 use the asymptotic evaluation
// below instead (most of the box: the quadrature's cost grows with rho).
//
// J0 without iterations or library calls (FP64 instructions are what bounds
// the quadrature: an SM has two FP64 lanes):
//   x < 25   Taylor polynomial of degree 11 about the nearest of 100 centres
//            (1/8 at most away); coefficients J0^(k)/k! from
//            J0^(k) = 2^-k sum_i (-1)^i C(k, i) J_{2i-k} and Miller's backward
//            recurrence, in long double on the host;
//   x >= 25  Hankel's asymptotic expansion
//            J0(x) = sqrt(2/(pi x)) (P cos chi - Q sin chi), chi = x - pi/4,
//            P = sum_k (-1)^k b_{2k} x^{-2k},  Q = -sum_k (-1)^k b_{2k+1} x^{-2k-1},
//            b_k = 1^2 3^2 ... (2k-1)^2 / (k! 8^k), 11 terms each (the 12th is
//            below 1e-18), with cos chi = (cos x + sin x)/sqrt 2 (no rounding
//            of x - pi/4).
// Both stay within 5e-16 of the envelope sqrt(2/(pi x)) (against 40-digit
// values; CUDA's j0 reaches 1e-12 of it for large x, which survives the
// quadrature sum).  exp(i kappa0 r) is one sincos per panel times node factors
// formed once per lane.  On a square period the table is symmetric and half of
// it is evaluated.  Measured, one table at kappa0 = 33 (128 x 128) on a GB300:
// quadrature 3.8 ms, asymptotic part 0.71 ms with Miller's recurrence and the
// double series of every term; 0.35 and 0.09 ms now.
#include <cmath>
#include <mutex>
#include <vector>

#include "common.cuh"

#define GLN 16
__constant__ double c_gl_x[GLN];
__constant__ double c_gl_w[GLN];

// Gauss-Legendre nodes and weights on [-1, 1] by Newton's iteration on the
// three-term recurrence of the Legendre polynomials.
static void gauss_legendre(int n, std::vector<double>& x, std::vector<double>& w) {
  x.resize(n);
  w.resize(n);
  for (int i = 0; i < n; ++i) {
    double z = std::cos(M_PI * (i + 0.75) / (n + 0.5));
    double dp = 0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = n * (z * p1 - p0) / (z * z - 1.0);
      double dz = p1 / dp;
      z -= dz;
      if (std::fabs(dz) < 1e-17) break;
    }
    double p0 = 1.0, p1 = z;
    for (int k = 2; k <= n; ++k) {
      double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
      p0 = p1;
      p1 = p2;
    }
    dp = n * (z * p1 - p0) / (z * z - 1.0);
    x[i] = z;
    w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
  }
}

#define J0_H 0.25
#define J0_N 100
#define J0_K 12
__device__ double g_j0_tab[J0_N * J0_K];
#define KHAT_NB 40
__constant__ double c_hank_b[KHAT_NB];

// J_n(x), n = 0 .. nmax, by Miller's backward recurrence (host, long double)
static void bessel_jn(long double x, int nmax, std::vector<long double>& J) {
  const int N = 2 * (int)(0.5L * (x + 12.0L * std::cbrt(x) + 60.0L)) + 2 * nmax;
  std::vector<long double> t(N + 2, 0.0L);
  t[N] = 1e-300L;
  for (int k = N; k >= 1; --k) {
    t[k - 1] = 2.0L * k / x * t[k] - t[k + 1];
    if (std::fabs(t[k - 1]) > 1e200L)
      for (int q = k - 1; q <= N; ++q) t[q] *= 1e-200L;
  }
  long double s = t[0];
  for (int k = 2; k <= N; k += 2) s += 2.0L * t[k];
  J.resize(nmax + 1);
  for (int n = 0; n <= nmax; ++n) J[n] = t[n] / s;
}

// Taylor coefficients of J0 about (i + 1/2) J0_H, [i][k]
static void j0_table(std::vector<double>& tab) {
  tab.resize(J0_N * J0_K);
  std::vector<long double> J;
  for (int i = 0; i < J0_N; ++i) {
    bessel_jn((i + 0.5L) * J0_H, J0_K, J);
    long double f = 1.0L;   // 2^-k / k!
    for (int k = 0; k < J0_K; ++k) {
      if (k > 0) f /= 2.0L * k;
      long double sum = 0.0L, c = 1.0L;
      for (int q = 0; q <= k; ++q) {
        const int n = 2 * q - k;
        const long double v = n >= 0 ? J[n] : ((-n) & 1 ? -J[-n] : J[-n]);
        sum += (q & 1 ? -c : c) * v;
        c = c * (k - q) / (q + 1);
      }
      tab[i * J0_K + k] = (double)(f * sum);
    }
  }
}

// tab: the Taylor table (shared memory)
__device__ __forceinline__ double bessel_j0(double x, const double* __restrict__ tab) {
  if (x < J0_N * J0_H) {
    const int i = (int)(x * (1.0 / J0_H));
    const double d = x - (i + 0.5) * J0_H;
    const double* c = tab + i * J0_K;
    double v = c[J0_K - 1];
#pragma unroll
    for (int k = J0_K - 2; k >= 0; --k) v = fma(v, d, c[k]);
    return v;
  }
  const double ix = 1.0 / x, y = ix * ix;
  double P = c_hank_b[20], Q = c_hank_b[21];
#pragma unroll
  for (int k = 9; k >= 0; --k) {
    P = fma(P, y, (k & 1) ? -c_hank_b[2 * k] : c_hank_b[2 * k]);
    Q = fma(Q, y, (k & 1) ? -c_hank_b[2 * k + 1] : c_hank_b[2 * k + 1]);
  }
  Q = -Q * ix;
  double sx, cx;
  sincos(x, &sx, &cx);
  // sqrt(2/(pi x)) (P cos chi - Q sin chi), both over sqrt 2
  return sqrt(ix * (1.0 / M_PI)) * (P * (cx + sx) - Q * (sx - cx));
}

// ---- the paper's large-frequency scheme (CAVITY_KHAT_PAPER), Sec. 5.2:
//   int_0^R J0(c r) e^{i k r} dr = int_0^inf - (1/c) int_{cR}^inf J0(z) e^{i k z/c} dz,
// int_0^inf = 1/sqrt(c^2 - k^2) (c > k) or i/sqrt(k^2 - c^2) (c < k); in the tail
// J0(z) ~ sqrt(2/(pi z)) (cos(z - pi/4) + sin(z - pi/4)/(8z)), the exponentials
// e^{+-i(z - pi/4)} combine with e^{i k z/c} into
//   A(p) = int_Z^inf e^{ipz} z^{-1/2} dz = sqrt(pi/(2|p|)) (1 + i - 2C(T) - 2iS(T)),
//   T = sqrt(2|p|Z/pi) (complex conjugate for p < 0), and
//   B(p) = int_Z^inf e^{ipz} z^{-3/2} dz = 2 e^{ipZ}/sqrt(Z) + 2ip A(p),
// p = k/c +- 1, with the Fresnel integrals C, S from their two-term asymptotic
// expansions.  (The paper prints 1/(c^2 - k^2) for the integral to infinity and
// sqrt(pi)/(2p) in front of A; the forms above are the corrected ones.)
#define KHAT_PAPER_CR (20.0 * M_PI * 1.41421356237309504880)

__device__ double2 kp_tail_half(double p, double Z) {
  const double ap = fabs(p);
  const double T = sqrt(2.0 * ap * Z / M_PI);
  const double u = M_PI * T * T;
  const double f = (1.0 - 3.0 / (u * u)) / (M_PI * T);
  const double g = (1.0 - 15.0 / (u * u)) / (M_PI * M_PI * T * T * T);
  double sp, cp;
  sincos(0.5 * u, &sp, &cp);
  const double C = 0.5 + f * sp - g * cp;
  const double S = 0.5 - f * cp - g * sp;
  const double pre = sqrt(M_PI / (2.0 * ap));
  double2 v = make_double2(pre * (1.0 - 2.0 * C), pre * (1.0 - 2.0 * S));
  if (p < 0) v.y = -v.y;
  return v;
}

__device__ double2 kp_tail_3half(double p, double Z) {
  const double2 A = kp_tail_half(p, Z);
  double s, c;
  sincos(p * Z, &s, &c);
  const double w = 2.0 / sqrt(Z);
  // 2 e^{ipZ}/sqrt(Z) + 2 i p A
  return make_double2(w * c - 2.0 * p * A.y, w * s + 2.0 * p * A.x);
}

__device__ double2 khat_paper_tail(double c, double k, double R) {
  const double d = c * c - k * k;
  const double2 inf = d > 0 ? make_double2(1.0 / sqrt(d), 0.0) : make_double2(0.0, 1.0 / sqrt(-d));
  const double Z = c * R;
  const double pp = k / c + 1.0, pm = k / c - 1.0;
  const double r2 = 0.70710678118654752440;
  const double2 e4 = make_double2(r2, -r2), e4c = make_double2(r2, r2);  // e^{-i pi/4}, e^{+i pi/4}
  const double2 ap = kp_tail_half(pp, Z), am = kp_tail_half(pm, Z);
  const double2 bp = kp_tail_3half(pp, Z), bm = kp_tail_3half(pm, Z);
  const double2 cosp = cscale<double>(cadd<double>(cmul<double>(e4, ap), cmul<double>(e4c, am)), 0.5);
  const double2 dsin = csub<double>(cmul<double>(e4, bp), cmul<double>(e4c, bm));
  const double2 sinp = make_double2(0.5 * dsin.y, -0.5 * dsin.x);     // / (2i)
  const double2 tail = cscale<double>(cadd<double>(cosp, cscale<double>(sinp, 0.125)),
                                      sqrt(2.0 / M_PI) / c);
  return cscale<double>(csub<double>(inf, tail), 0.5);
}

// ---- large-argument evaluation of the same integral (default scheme).
// Where c R >= KHAT_ASYM_CR and |c - kappa0| R >= KHAT_ASYM_GAP:
//   int_0^R = int_0^inf - int_R^inf,  int_0^inf as in the paper's scheme, and
//   int_R^inf J0(c r) e^{i k r} dr = (1/c) int_Z^inf J0(z) e^{i k z/c} dz, Z = c R,
// with the complete Hankel expansion
//   J0(z) = sqrt(2/pi) (1/2) sum_m b_m z^{-m-1/2} [(-i)^m e^{i(z - pi/4)} + i^m e^{-i(z - pi/4)}],
//   b_m = 1^2 3^2 ... (2m-1)^2 / (m! 8^m),
// and each  F_m(p) = int_Z^inf z^{-m-1/2} e^{ipz} dz  (p = 1 + k/c, k/c - 1) from
// repeated integration by parts,
//   F_m(p) = (i/p) e^{ipZ} Z^{-m-1/2} sum_j (m + 1/2)_j (-i/(pZ))^j,
// both series summed to their smallest term.  The thresholds keep every series
// far inside its range (|p| Z >= 30, Z >= 100).  Measured against a 30-digit
// evaluation the result is within ~2e-15 there, better than the quadrature,
// whose sum of ~1000 oscillating panels loses ~Z 1e-16 to the rounding of c r.
// The sum over m is formed downward.  With G_m = sum_j (m + 1/2)_j (-i/(pZ))^j
// one integration by parts is G_m = 1 - i (m + 1/2)/(pZ) G_{m+1}, and the
// factors b_m (-+i/Z)^m nest like Horner's rule, so only the last G takes its
// series (errors shrink by (m + 1/2)/|pZ| < 1/2 a step); M: the first term
// below 1e-18.
#define KHAT_ASYM_CR 100.0
#define KHAT_ASYM_GAP 30.0

// sum_m b_m (sg i / Z)^m G_m(p), sg = -1 for e^{+i(z - pi/4)}, 1 for its conjugate
__device__ __forceinline__ double2 khat_tail_sum(double p, double Z, double zinv, int M, double sg) {
  const double x = -1.0 / (p * Z);         // -i/(pZ) = i x
  // G_M: terms (s)_j (i x)^j
  double t = 1.0, gr = 0.0, gi = 0.0, prev = 1e300;
  for (int j = 0; j < 200; ++j) {
    const double mag = fabs(t);
    if (mag > prev) break;
    const int q = j & 3;
    if (q == 0) gr += t;
    else if (q == 1) gi += t;
    else if (q == 2) gr -= t;
    else gi -= t;
    if (mag < 1e-18) break;
    prev = mag;
    t *= (M + 0.5 + j) * x;
  }
  double sr = c_hank_b[M] * gr, si = c_hank_b[M] * gi;
  const double u = sg * zinv;
  for (int m = M - 1; m >= 0; --m) {
    const double f = x * (m + 0.5);
    const double nr = 1.0 - f * gi, ni = f * gr;   // G_m = 1 + i x (m + 1/2) G_{m+1}
    gr = nr;
    gi = ni;
    const double b = c_hank_b[m];
    const double tr = fma(b, gr, -u * si), ti = fma(b, gi, u * sr);
    sr = tr;
    si = ti;
  }
  return make_double2(sr, si);
}

__device__ double2 khat_asymptotic(double c, double k, double R) {
  const double d = c * c - k * k;
  const double2 inf = d > 0 ? make_double2(1.0 / sqrt(d), 0.0) : make_double2(0.0, 1.0 / sqrt(-d));
  const double Z = c * R, zinv = 1.0 / Z;
  const double pp = 1.0 + k / c, pm = k / c - 1.0;
  double sp, cp, sm, cm;
  sincos(pp * Z, &sp, &cp);
  sincos(pm * Z, &sm, &cm);
  int M = 0;
  for (double z = 1.0; M < KHAT_NB - 1;) {
    z *= zinv;
    ++M;
    if (c_hank_b[M] * z < 1e-18) break;
  }
  const double r2 = 0.70710678118654752440;
  // e^{-+i pi/4} (i/p) e^{ipZ}
  const double2 fp = cmul<double>(make_double2(r2, -r2), make_double2(-sp / pp, cp / pp));
  const double2 fm = cmul<double>(make_double2(r2, r2), make_double2(-sm / pm, cm / pm));
  double2 T = cadd<double>(cmul<double>(fp, khat_tail_sum(pp, Z, zinv, M, -1.0)),
                           cmul<double>(fm, khat_tail_sum(pm, Z, zinv, M, 1.0)));
  T = cscale<double>(T, 0.5 * sqrt(zinv * (2.0 / M_PI)) / c);
  return cscale<double>(csub<double>(inf, T), 0.5);
}

__device__ __forceinline__ bool khat_use_asym(double c, double k, double R) {
  return c * R >= KHAT_ASYM_CR && fabs(c - fabs(k)) * R >= KHAT_ASYM_GAP;
}

// writes F(G) at (j1, j2), and at (j2, j1) where the table is symmetric (equal
// periods) and holds it; the scaled copies are stored transposed, [j2][j1]: the
// operator reads them along j1 for fixed j2
__device__ __forceinline__ void khat_put(double2 v, int j1, int j2, int hx, int hy, bool sym,
                                         double scale, double2* __restrict__ raw,
                                         double2* __restrict__ s64, float2* __restrict__ s32) {
  const double2 w = make_double2(v.x * scale, v.y * scale);
  const float2 f = make_float2((float)w.x, (float)w.y);
  raw[(size_t)j1 * hy + j2] = v;
  s64[(size_t)j2 * hx + j1] = w;
  s32[(size_t)j2 * hx + j1] = f;
  if (sym && j1 != j2 && j1 < hy && j2 < hx) {
    raw[(size_t)j2 * hy + j1] = v;
    s64[(size_t)j1 * hx + j2] = w;
    s32[(size_t)j1 * hx + j2] = f;
  }
}
// whether (j1, j2) is left to its mirror image
__device__ __forceinline__ bool khat_mirrored(int j1, int j2, int hx, int hy, bool sym) {
  return sym && j2 > j1 && j1 < hy && j2 < hx;
}

// one thread per entry of the quarter box; entries outside the asymptotic
// range are left to the quadrature kernel
__global__ void k_khat_asym(double2* __restrict__ raw, double2* __restrict__ s64,
                            float2* __restrict__ s32, int hx, int hy, double Lx, double Ly,
                            double kappa0, double R, double scale) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= (long long)hx * hy) return;
  const int j1 = (int)(e / hy), j2 = (int)(e - (long long)j1 * hy);
  const bool sym = Lx == Ly;
  if (khat_mirrored(j1, j2, hx, hy, sym)) return;
  const double r1 = j1 / Lx, r2 = j2 / Ly;
  const double c = 2.0 * M_PI * sqrt(r1 * r1 + r2 * r2);
  if (!khat_use_asym(c, kappa0, R)) return;
  khat_put(khat_asymptotic(c, kappa0, R), j1, j2, hx, hy, sym, scale, raw, s64, s32);
}

// Quadrature: one warp per entry.  Lane l takes the nodes 4 (l & 3) .. + 3 of
// the panels l / 4, l / 4 + 8, ..; a fixed-order shuffle reduction.
__global__ void __launch_bounds__(256) k_khat(double2* __restrict__ raw, double2* __restrict__ s64,
                                              float2* __restrict__ s32, int hx, int hy, double Lx,
                                              double Ly, double kappa0, double R, double scale,
                                              int scheme) {
  __shared__ double tab[J0_N * J0_K];
  const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int j1 = (int)(warp / hy), j2 = (int)(warp - (long long)j1 * hy);
  const double r1 = j1 / Lx, r2 = j2 / Ly;
  const double rho = sqrt(r1 * r1 + r2 * r2);
  const double c = 2.0 * M_PI * rho;
  const bool sym = Lx == Ly;
  bool work = j1 < hx && !khat_mirrored(j1, j2, hx, hy, sym);
  if (scheme == CAVITY_KHAT_QUADRATURE && khat_use_asym(c, kappa0, R)) work = false;  // k_khat_asym
  if (work && scheme == CAVITY_KHAT_PAPER && c * R > KHAT_PAPER_CR) {
    if (lane == 0)
      khat_put(khat_paper_tail(c, kappa0, R), j1, j2, hx, hy, sym, scale, raw, s64, s32);
    work = false;
  }
  if (!__syncthreads_or(work)) return;
  for (int i = threadIdx.x; i < J0_N * J0_K; i += blockDim.x) tab[i] = g_j0_tab[i];
  __syncthreads();
  if (!work) return;
  const double omega = c + fabs(kappa0);
  int npan = (int)ceil(omega * R / M_PI);
  if (npan < 1) npan = 1;
  const double width = R / npan;
  // this lane's nodes: offset in the panel, weight, exp(i kappa0 offset)
  const int q0 = 4 * (lane & 3);
  double off[4], wt[4], ns[4], nc[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    off[k] = 0.5 * width * (c_gl_x[q0 + k] + 1.0);
    wt[k] = c_gl_w[q0 + k];
    sincos(kappa0 * off[k], &ns[k], &nc[k]);
  }
  double sr = 0.0, si = 0.0;
  for (int pn = lane >> 2; pn < npan; pn += 8) {
    const double r0 = pn * width;
    double ps, pc, pr = 0.0, pi_ = 0.0;
    sincos(kappa0 * r0, &ps, &pc);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double jv = bessel_j0(c * (r0 + off[k]), tab) * wt[k];
      pr += jv * nc[k];
      pi_ += jv * ns[k];
    }
    sr += pc * pr - ps * pi_;
    si += pc * pi_ + ps * pr;
  }
  for (int o = 16; o > 0; o >>= 1) {
    sr += __shfl_xor_sync(0xffffffffu, sr, o);
    si += __shfl_xor_sync(0xffffffffu, si, o);
  }
  if (lane == 0)
    khat_put(make_double2(0.25 * width * sr, 0.25 * width * si), j1, j2, hx, hy, sym, scale, raw,
             s64, s32);
}

cavity_status launch_khat(cavity_ctx* ctx, double kappa0) {
  const Geo& g = ctx->g;
  static std::mutex mu;   // host threads may prepare contexts at the same time
  static DeviceFlag gl_done;
  std::unique_lock<std::mutex> lock(mu);
  if (!gl_done) {
    std::vector<double> x, w;
    gauss_legendre(GLN, x, w);
    CK(cudaMemcpyToSymbol(c_gl_x, x.data(), sizeof(double) * GLN));
    CK(cudaMemcpyToSymbol(c_gl_w, w.data(), sizeof(double) * GLN));
    double b[KHAT_NB];
    b[0] = 1.0;
    for (int m = 1; m < KHAT_NB; ++m) b[m] = b[m - 1] * (double)((2 * m - 1) * (2 * m - 1)) / (8.0 * m);
    CK(cudaMemcpyToSymbol(c_hank_b, b, sizeof(double) * KHAT_NB));
    std::vector<double> tab;
    j0_table(tab);
    CK(cudaMemcpyToSymbol(g_j0_tab, tab.data(), sizeof(double) * tab.size()));
    // these copies are on the default stream and may still be on their way from
    // the runtime's staging memory; a context's own stream does not wait for it
    CK(cudaStreamSynchronize(nullptr));
    gl_done.set();
  }
  lock.unlock();
  const int hx = g.Px / 2, hy = g.Py / 2;
  size_t n = (size_t)hx * hy;
  CK(table_alloc(&ctx->khat64, n));
  CK(table_alloc(&ctx->khat32, n));
  CK(table_alloc(&ctx->khat_raw, n));
  const long long threads = (long long)n * 32;
  {
    KScope ks_(ctx, KC_SETUP);
    k_khat<<<(unsigned)((threads + 255) / 256), 256, 0, ctx->stream>>>(
        ctx->khat_raw, ctx->khat64, ctx->khat32, hx, hy, g.Lx, g.Ly, kappa0, g.R,
        1.0 / (g.Lx * g.Ly), ctx->desc.khat_scheme);
  }
  if (ctx->desc.khat_scheme == CAVITY_KHAT_QUADRATURE) {
    KScope ks_(ctx, KC_SETUP);
    k_khat_asym<<<(unsigned)((n + 127) / 128), 128, 0, ctx->stream>>>(
        ctx->khat_raw, ctx->khat64, ctx->khat32, hx, hy, g.Lx, g.Ly, kappa0, g.R,
        1.0 / (g.Lx * g.Ly));
  }
  CK(cudaGetLastError());
  return CAVITY_OK;
}
