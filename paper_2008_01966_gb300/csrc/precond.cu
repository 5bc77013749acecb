// Block-diagonal preconditioner of the aperture system (EJ1)/(uT1).
//
// The coefficients E1^{mn}, E2^{mn}, E3^{mn} of one mode (m, n) are coupled
// by the cavity part (row 3 and the E3 columns of rows 1, 2) and by the
// diagonal entries of the three TBC integrals I1, I2, I3 of Sec. 5.1.  Those
// diagonals are evaluated exactly under the same discrete rule as the
// operator itself:
//     I^{mn}_{mn} = sum_{j1, j2} Ax(m, j1) F(G)(j1, j2) Ay(n, j2) / (Lx Ly),
//     Ax(m, j1) = X(m, j1) Phi(j1, m),
// with X the trapezoid projection of the torus Fourier mode exp(2 pi i j1 x/Lx)
// onto cos/sin(m pi x/a) and Phi the exact basis transform of Sec. 5.2.  Both
// factors are symmetric or antisymmetric about the middle of the side together,
// so Ax is real and even in j1: the sums run over j1, j2 >= 0 as two products
// of real factors with the complex table.  Their FP64 operations are what
// bounds them (two lanes per SM); outputs are spread over tiles of 16 x 16 so
// that small grids fill the machine.  The trapezoid sums X are geometric
// progressions in closed form.  Measured at 128 x 128 on a GB300 (Ax, both
// axes; the two products): 0.48, 0.46 and 0.65 ms with term-by-term sums and
// complex factors; 0.07, 0.07 and 0.07 ms now.  The
// 3x3 blocks (2x2 / 1x1 where a component is absent) are inverted once per
// (kappa0, eps) and applied as a right preconditioner in GMRES.  Only the
// iteration count depends on it, never the solution.
#include "common.cuh"

// Trapezoid sum of a geometric progression (weights 1/2, 1, .., 1, 1/2 over
// p = 0..N) with the ratio z = exp(i pi q / P), N = P / pad:
//   (i/2) cot(pi q / 2P) (1 - z^N),  z^N = exp(i pi q / pad);  N at q = 0.
// q is an integer, so every angle is exact.
__device__ __forceinline__ double2 pc_prog(int q, int P, int pad) {
  if (q == 0) return make_double2((double)(P / pad), 0.0);
  double s, c, es, ec;
  sincospi((double)q / (2.0 * P), &s, &c);
  sincospi((double)(q % (2 * pad)) / pad, &es, &ec);
  const double ct = 0.5 * c / s;
  return make_double2(ct * es, ct * (1.0 - ec));
}

// Ax[kind][m][j], 0 <= j < P/2, doubled for j > 0 (the sum over +-j)
__global__ void k_pc_ax(double* __restrict__ out, int nint, int Pn, double side, int pad) {
  const int kind = blockIdx.z;  // 0 cos, 1 sin
  const int m = blockIdx.y, hp = Pn / 2;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < hp; j += gridDim.x * blockDim.x) {
    double r = 0;
    if (!(kind == 1 && m == 0)) {
      // cos, sin(m pi p / N) exp(2 pi i j p / P) as progressions of 2 j +- pad m
      const double2 gp = pc_prog(2 * j + pad * m, Pn, pad), gm = pc_prog(2 * j - pad * m, Pn, pad);
      const double w = 0.5 * side / nint;
      const long long sh = (long long)(pad / 2) * m;
      const double2 em = eps_d(j - sh, side, pad), ep = eps_d(j + sh, side, pad);
      double2 X, phi;
      if (kind == 0) {
        X = make_double2(w * (gp.x + gm.x), w * (gp.y + gm.y));
        phi = make_double2(0.5 * (em.x + ep.x), 0.5 * (em.y + ep.y));
      } else {
        X = make_double2(w * (gp.y - gm.y), -w * (gp.x - gm.x));            // /(2i)
        phi = make_double2(0.5 * (em.y - ep.y), -0.5 * (em.x - ep.x));
      }
      r = (j > 0 ? 2.0 : 1.0) * (X.x * phi.x - X.y * phi.y);
    }
    out[((size_t)kind * nint + m) * hp + j] = r;
  }
}

// C[i][j] = sum_k A[i][k] B[j][k], one of A, B real (double), the other complex;
// 16 x 16 outputs per block of 256 threads, k-tiles of 32.  grid (ceil(Nc / 16),
// ceil(Mr / 16), batch); batch element f reads A + ao[f], B + bo[f] and writes
// C + f cs.
struct PcOff {
  long long a[3], b[3], cs;
};
template <typename TA, typename TB>
__global__ void __launch_bounds__(256) k_pc_gemm(const TA* __restrict__ A, int lda,
                                                 const TB* __restrict__ B, int ldb,
                                                 double2* __restrict__ C, int ldc, int Mr, int Nc,
                                                 int K, PcOff off) {
  __shared__ TA as[16][33];
  __shared__ TB bs[16][33];
  const int f = blockIdx.z, t = threadIdx.x, ti = t >> 4, tj = t & 15;
  const int i0 = blockIdx.y * 16, j0 = blockIdx.x * 16;
  A += off.a[f];
  B += off.b[f];
  double sx = 0, sy = 0;
  for (int k0 = 0; k0 < K; k0 += 32) {
    for (int e = t; e < 512; e += 256) {
      const int r = e >> 5, k = e & 31;
      const bool kin = k0 + k < K;
      as[r][k] = (kin && i0 + r < Mr) ? A[(size_t)(i0 + r) * lda + k0 + k] : TA{};
      bs[r][k] = (kin && j0 + r < Nc) ? B[(size_t)(j0 + r) * ldb + k0 + k] : TB{};
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
      if constexpr (std::is_same<TA, double>::value) {
        sx = fma(as[ti][k], bs[tj][k].x, sx);
        sy = fma(as[ti][k], bs[tj][k].y, sy);
      } else {
        sx = fma(bs[tj][k], as[ti][k].x, sx);
        sy = fma(bs[tj][k], as[ti][k].y, sy);
      }
    }
    __syncthreads();
  }
  if (i0 + ti < Mr && j0 + tj < Nc)
    C[f * off.cs + (size_t)(i0 + ti) * ldc + j0 + tj] = make_double2(sx, sy);
}

__device__ void inv3(double2 A[3][3], double2 Bi[3][3]) {
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) Bi[r][c] = make_double2(r == c ? 1.0 : 0.0, 0.0);
  for (int k = 0; k < 3; ++k) {
    int piv = k;
    double best = cabs2<double>(A[k][k]);
    for (int r = k + 1; r < 3; ++r)
      if (cabs2<double>(A[r][k]) > best) { best = cabs2<double>(A[r][k]); piv = r; }
    if (piv != k)
      for (int c = 0; c < 3; ++c) {
        double2 t = A[k][c]; A[k][c] = A[piv][c]; A[piv][c] = t;
        t = Bi[k][c]; Bi[k][c] = Bi[piv][c]; Bi[piv][c] = t;
      }
    double2 inv = cdiv<double>(make_double2(1, 0), A[k][k]);
    for (int c = 0; c < 3; ++c) { A[k][c] = cmul<double>(A[k][c], inv); Bi[k][c] = cmul<double>(Bi[k][c], inv); }
    for (int r = 0; r < 3; ++r) {
      if (r == k) continue;
      double2 f = A[r][k];
      for (int c = 0; c < 3; ++c) {
        A[r][c] = csub<double>(A[r][c], cmul<double>(f, A[k][c]));
        Bi[r][c] = csub<double>(Bi[r][c], cmul<double>(f, Bi[k][c]));
      }
    }
  }
}

__global__ void k_pc_blocks(const double2* __restrict__ dd, const double2* __restrict__ top,
                            double2* __restrict__ pinv, float2* __restrict__ pinv32, int nx, int ny,
                            int n1, int n2, int nap, double a, double b, double h, double k2) {
  const int m = blockIdx.y;
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= ny) return;
  const int N = ny - 1;
  const double2* d1 = dd + ((size_t)0 * nx + m) * (ny + 1);
  const double2* d2 = dd + ((size_t)1 * nx + m) * (ny + 1);
  const double2* d3 = dd + ((size_t)2 * nx + m) * (ny + 1);
  const double mx = m * M_PI / a, nyv = n * M_PI / b;
  const double ab = a * b;
  const double sq = h / (m == 0 ? ab / 2 : ab / 4), sc = h / (n == 0 ? ab / 2 : ab / 4);
  double2 A[3][3];
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) A[r][c] = make_double2(r == c ? 1.0 : 0.0, 0.0);
  const bool has1 = n >= 1, has2 = m >= 1, has3 = m >= 1 && n >= 1;
  const int i1 = m * N + (n - 1), i2 = n1 + (m - 1) * (N + 1) + n;
  const int i3 = n1 + n2 + (m - 1) * N + (n - 1);
  if (has1) {
    double2 tb = csub<double>(cscale<double>(d1[n], k2), cscale<double>(d3[n], 2 * nyv * nyv));
    A[0][0] = cadd<double>(make_double2(-1.0 + top[i1].x, top[i1].y), cscale<double>(tb, sq));
  }
  if (has2) {
    double2 tb = csub<double>(cscale<double>(d2[n], k2), cscale<double>(d3[n], 2 * mx * mx));
    A[1][1] = cadd<double>(make_double2(-1.0 + top[i2].x, top[i2].y), cscale<double>(tb, sc));
  }
  if (has3) {
    A[0][1] = cscale<double>(d3[n], sq * 2 * nyv * mx);
    A[0][2] = make_double2(mx * h + top[nap + i1].x, top[nap + i1].y);
    A[1][0] = cscale<double>(d3[n], sc * 2 * mx * nyv);
    A[1][2] = make_double2(nyv * h + top[nap + i2].x, top[nap + i2].y);
    A[2][0] = make_double2(mx * h, 0);
    A[2][1] = make_double2(nyv * h, 0);
    A[2][2] = make_double2(-1.0 + top[i3].x, top[i3].y);
  }
  double2 Bi[3][3];
  inv3(A, Bi);
  double2* o = pinv + ((size_t)m * ny + n) * 9;
  float2* o32 = pinv32 + ((size_t)m * ny + n) * 9;
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) {
      o[r * 3 + c] = Bi[r][c];
      o32[r * 3 + c] = make_float2((float)Bi[r][c].x, (float)Bi[r][c].y);
    }
}

cavity_status launch_precond(cavity_ctx* ctx) {
  const Geo& g = ctx->g;
  const int hx = g.Px / 2, hy = g.Py / 2;
  size_t nax = (size_t)2 * g.nx * hx, nay = (size_t)2 * g.ny * hy;
  size_t nT = (size_t)2 * g.nx * hy, nd = (size_t)3 * g.nx * (g.ny + 1);
  size_t need = sizeof(double) * (nax + nay) + sizeof(double2) * (nT + nd);
  CKS(ensure_ws(ctx, &ctx->ws2, &ctx->ws2_bytes, need));
  double2* T = (double2*)ctx->ws2;
  double2* dd = T + nT;
  double* ax = (double*)(dd + nd);
  double* ay = ax + nax;
  CK(table_alloc(&ctx->pinv64, 9 * (size_t)g.nx * g.ny));
  CK(table_alloc(&ctx->pinv32, 9 * (size_t)g.nx * g.ny));
  cudaStream_t st = ctx->stream;
  {
    KScope ks_(ctx, KC_SETUP);
    k_pc_ax<<<dim3((hx + 127) / 128, g.nx, 2), 128, 0, st>>>(ax, g.nx, g.Px, g.a, g.padx);
  }
  {
    KScope ks_(ctx, KC_SETUP);
    k_pc_ax<<<dim3((hy + 127) / 128, g.ny, 2), 128, 0, st>>>(ay, g.ny, g.Py, g.b, g.pady);
  }
  {
    // T[xk][m][j2] = sum_j1 Ax[xk][m][j1] F(G)(j1, j2)   (table stored [j2][j1])
    KScope ks_(ctx, KC_SETUP);
    k_pc_gemm<double, double2><<<dim3((hy + 15) / 16, (2 * g.nx + 15) / 16, 1), 256, 0, st>>>(
        ax, hx, ctx->khat64, hx, T, hy, 2 * g.nx, hy, hx, PcOff{{0, 0, 0}, {0, 0, 0}, 0});
  }
  {
    // d[f][m][n] = sum_j2 T[xk][m][j2] Ay[yk][n][j2];  f: 0 cs, 1 sc, 2 cc
    const long long tx = (long long)g.nx * hy, ty = (long long)g.ny * hy;
    KScope ks_(ctx, KC_SETUP);
    k_pc_gemm<double2, double><<<dim3((g.ny + 15) / 16, (g.nx + 15) / 16, 3), 256, 0, st>>>(
        T, hy, ay, hy, dd, g.ny + 1, g.nx, g.ny, hy,
        PcOff{{0, tx, 0}, {ty, 0, 0}, (long long)g.nx * (g.ny + 1)});
  }
  {
    KScope ks_(ctx, KC_SETUP);
    k_pc_blocks<<<dim3((g.ny + 127) / 128, g.nx), 128, 0, st>>>(
        dd, ctx->top64, ctx->pinv64, ctx->pinv32, g.nx, g.ny, g.n1, g.n2, g.nap, g.a, g.b, g.h,
        2.0 * ctx->kappa0 * ctx->kappa0);
  }
  CK(cudaGetLastError());
  return CAVITY_OK;
}

// y = (block diagonal)^{-1} x at mode pair mn; pm: order of x
template <typename T>
__device__ __forceinline__ void pc_mode(const C<T>* __restrict__ xd, C<T>* __restrict__ yd, int mn,
                                        const C<T>* __restrict__ pinv, int ny, int n1, int n2,
                                        const ParityMap& pm) {
  const int lny = __ffs(ny) - 1;                 // ny is a power of two
  const int m = mn >> lny, n = mn & (ny - 1);
  const int N = ny - 1;
  const bool has1 = n >= 1, has2 = m >= 1, has3 = m >= 1 && n >= 1;
  const int i1 = m * N + (n - 1), i2 = n1 + (m - 1) * (N + 1) + n;
  const int i3 = n1 + n2 + (m - 1) * N + (n - 1);
  C<T> v[3] = {mk<T>(0, 0), mk<T>(0, 0), mk<T>(0, 0)};
  if (has1) v[0] = xd[pm.on ? pm.e1(m, n) : i1];
  if (has2) v[1] = xd[pm.on ? pm.e2(m, n) : i2];
  if (has3) v[2] = xd[pm.on ? pm.e3(m, n) : i3];
  const C<T>* B = pinv + (size_t)mn * 9;
  C<T> r[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    r[a] = cmul<T>(B[a * 3 + 0], v[0]);
    r[a] = cadd<T>(r[a], cmul<T>(B[a * 3 + 1], v[1]));
    r[a] = cadd<T>(r[a], cmul<T>(B[a * 3 + 2], v[2]));
  }
  if (has1) yd[i1] = r[0];
  if (has2) yd[i2] = r[1];
  if (has3) yd[i3] = r[2];
}

// y = (block diagonal)^{-1} x for ndir vectors
template <typename T>
__global__ void k_pc_apply(const C<T>* __restrict__ x, long long xs, C<T>* __restrict__ y,
                           long long ys, const C<T>* __restrict__ pinv, int nx, int ny, int n1,
                           int n2, int nap, int ndir, ParityMap pm) {
  long long gid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long per = (long long)nx * ny;
  if (gid >= per * ndir) return;
  const int d = (int)(gid / per);
  pc_mode<T>(x + (size_t)d * xs, y + (size_t)d * ys, (int)(gid - (long long)d * per), pinv, ny, n1,
             n2, pm);
}
// the same for the columns of several groups; grid (ceil(nx ny / 256), ncol)
__global__ void k_pc_groups(PcCols cols, float2* __restrict__ y, const float2* __restrict__ pinv,
                            int nmode, int ny, int n1, int n2, int nap, ParityMap pm) {
  const int c = blockIdx.y, mn = blockIdx.x * blockDim.x + threadIdx.x;
  if (mn >= nmode) return;
  int g = 0;
  while (g + 1 < cols.n && cols.first[g + 1] <= c) ++g;
  pc_mode<float>(cols.src[g] + (size_t)(c - cols.first[g]) * nap, y + (size_t)c * nap, mn, pinv, ny,
                 n1, n2, pm);
}

template <typename T>
cavity_status launch_precond_apply(cavity_ctx* ctx, int ndir, const C<T>* x, C<T>* y,
                                   long long xs, long long ys, const ParityMap& pm) {
  if (xs < 0) xs = ctx->g.nap;
  if (ys < 0) ys = ctx->g.nap;
  const Geo& g = ctx->g;
  const C<T>* pinv;
  if (sizeof(T) == 8) pinv = (const C<T>*)ctx->pinv64;
  else pinv = (const C<T>*)ctx->pinv32;
  long long tot = (long long)g.nx * g.ny * ndir;
  {
    KScope ks_(ctx, KC_PRECOND);
    const int eb = elem_block(tot);
    k_pc_apply<T><<<(unsigned)((tot + eb - 1) / eb), eb, 0, ctx->stream>>>(x, xs, y, ys, pinv, g.nx,
        g.ny, g.n1, g.n2, g.nap, ndir, pm);
  }
  CK(cudaGetLastError());
  // two-level variant (FP32 inner solves of the mixed path): the coarse
  // unknowns take the exact solve of the coarse block instead
  if constexpr (std::is_same<T, float>::value) CKS(coarse_correct(ctx, ndir, x, xs, y, ys));
  return CAVITY_OK;
}

template cavity_status launch_precond_apply<double>(cavity_ctx*, int, const double2*, double2*,
                                                    long long, long long, const ParityMap&);
template cavity_status launch_precond_apply<float>(cavity_ctx*, int, const float2*, float2*,
                                                   long long, long long, const ParityMap&);

cavity_status launch_precond_groups(cavity_ctx* ctx, int ncol, const PcCols& cols, float2* y,
                                    const ParityMap& pm) {
  const Geo& g = ctx->g;
  if (ctx->opt[CAVITY_OPT_COARSE_MODES] > 0) {   // the coarse level works group by group
    for (int q = 0; q < cols.n; ++q) {
      const int n = (q + 1 < cols.n ? cols.first[q + 1] : ncol) - cols.first[q];
      CKS(launch_precond_apply<float>(ctx, n, cols.src[q], y + (size_t)cols.first[q] * g.nap, g.nap,
                                      g.nap, pm));
    }
    return CAVITY_OK;
  }
  KScope ks_(ctx, KC_PRECOND);
  k_pc_groups<<<dim3((g.nx * g.ny + 255) / 256, ncol), 256, 0, ctx->stream>>>(
      cols, y, ctx->pinv32, g.nx * g.ny, g.ny, g.n1, g.n2, g.nap, pm);
  CK(cudaGetLastError());
  return CAVITY_OK;
}
