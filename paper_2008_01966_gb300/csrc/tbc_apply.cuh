// The aperture operator of (EJ1)/(uT1): the cavity (local) part and the TBC
// part whose singular integrals follow Sec. 5 (discrete rule: periodised FFT
// convolution with the exact transform of the truncated basis, the kernel
// table F(G), inverse transform on the torus grid, trapezoid outer rule).
//
// For each right-hand side the TBC needs three convolution-projections,
//   U1 = <cs_mn, G*u1>,  U2 = <sc_mn, G*u2>,  W = <cc_mn, G*w>,
// u1 = sum E1 cs, u2 = sum E2 sc, w = div_Gamma(z x E) = sum (k2 pi/b) E1 cc -
// sum (k1 pi/a) E2 cc (Sec. 5.1 reduces every coefficient to I1, I2, I3).
// E1 is a sine series in x2 and E2 one in x1: each vanishes on the two edges
// across which w differentiates it, so the transform of the truncated w is
// exactly
//   F(w)(xi) = 2 pi i (xi2 F(E1)(xi) - xi1 F(E2)(xi)),
// and only E1 and E2 take the basis transform: pass A does 2/3 and pass B 3/4
// of the operations of three.  Both FP64 (two lanes per SM) and pair arithmetic
// (6 to 25 FP32 instructions per operation) are bound by operations; operator
// on one GB300, before and after: FP64 256 x 256, 6 vectors 6.43 -> 5.00 ms,
// 512 x 512, 4 vectors 18.5 -> 14.2 ms, 1024 x 1024, 2 vectors 41.9 -> 32.0 ms;
// pair, the same, 2.97 -> 2.34, 6.33 -> 5.07, 21.2 -> 17.2 ms (before the pair
// type's own line shape, df64.cuh).
// Four passes of batched line transforms in shared memory:
//   A  (rows k1)   basis transform of E1, E2 along x2: FFT convolution of the
//                  mirrored coefficients with the 1-D kernel E(nu) of F(F)
//   B  (cols j2)   basis transform along x1, w from it, all three fields times
//                  F(G)/(Lx Ly), inverse DFT along x1 at the nodes p = 0..Nx
//   C  (rows p)    inverse DFT along x2 at q = 0..Ny, trapezoid projection
//                  onto cos/sin(n pi q/Ny) (an extended FFT of length 2Ny)
//   D  (cols n)    trapezoid projection along x1 (extended FFT of length 2Nx)
// and a final elementwise pass adds the local part of (EJ1)/(uT1).
// Templated on the arithmetic type: FP64 for the FP64 path, pair-of-FP32 for the
// residuals of the mixed path.  Every pass kernel is instantiated per grid size
// so that its line transforms have compile-time lengths; tbc.cu instantiates the
// FP64 operator, tbc_df*.cu the pair-of-FP32 one.  The FP32 operator of the
// mixed path's inner iterations has passes of its own (tbc_f32.cu).
#pragma once
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "fft.cuh"

struct TbcP {
  int nx, ny, M, N, Px, Py, lPx, lPy, lnx, lny, nap, n1, n2;
  double a, b, h, k2x2;  // k2x2 = 2 kappa0^2
  double pia, pib, ab;   // pi / a, pi / b, a b
  double wy, wx;         // trapezoid weights / 2: b / (2 ny), a / (2 nx)
  int twlog;
};

static TbcP make_params(const cavity_ctx* ctx) {
  const Geo& g = ctx->g;
  TbcP p;
  p.nx = g.nx; p.ny = g.ny; p.M = g.M; p.N = g.N; p.Px = g.Px; p.Py = g.Py;
  p.lPx = g.lPx; p.lPy = g.lPy; p.lnx = g.lnx; p.lny = g.lny;
  p.nap = g.nap; p.n1 = g.n1; p.n2 = g.n2;
  p.a = g.a; p.b = g.b; p.h = g.h; p.k2x2 = 2.0 * ctx->kappa0 * ctx->kappa0;
  p.pia = M_PI / g.a; p.pib = M_PI / g.b; p.ab = g.a * g.b;
  p.wy = 0.5 * g.b / g.ny; p.wx = 0.5 * g.a / g.nx;
  p.twlog = ilog2(ctx->TW);
  return p;
}

template <typename T> __device__ __forceinline__ C<T> czero() { return mk<T>(0, 0); }

// Lines per CTA: enough lines that a pass of the longest transform in the
// kernel occupies the CTA's threads (nlong = that length).
template <typename T> __host__ __device__ constexpr int lines_per_cta(int nlong) {
  return fft_tpl<T>(nlong) >= FftE<T>::THREADS ? 1 : FftE<T>::THREADS / fft_tpl<T>(nlong);
}
// threads of a CTA of passes A and B: at 4096 points, where shared memory holds
// one CTA per SM, both lines of a pair side by side
template <typename T> __host__ __device__ constexpr int pair_threads(int n) {
  return n < 4096 ? FftE<T>::THREADS : 2 * FftE<T>::THREADS;
}
// passes A and B hold two lines (parities r = 0, 1) per row / column
template <typename T> __host__ __device__ constexpr int pairs_per_cta(int n) {
  return 2 * fft_tpl<T>(n) >= FftE<T>::THREADS ? 1 : FftE<T>::THREADS / (2 * fft_tpl<T>(n));
}
// These are the most lines of a CTA; a launch whose grid would not give every
// SM two CTAs takes fewer (halved until it does, with the threads to match):
// an SM has two FP64 lanes, so a 32 x 32 grid in 16 CTAs of eight columns used
// a tenth of the machine (operator on one FP64 vector at 32 x 32: 125 us,
// 164 us with full CTAs).  lL: log2 of the lines (or pairs) of a CTA.
struct CtaLines {
  int lL, threads;
  unsigned blocks(int lines) const { return (unsigned)((lines + (1 << lL) - 1) >> lL); }
};
inline CtaLines cta_lines(int lL_max, int per_line, int tpl, int most, long long lines,
                          long long batch) {
  const long long want = 2 * sm_count();
  int lL = lL_max;
  while (lL > 0 && ((lines + (1 << lL) - 1) >> lL) * batch < want) --lL;
  return CtaLines{lL, std::min(most, std::max(32, (per_line << lL) * tpl))};
}
// registers: the pass kernels run two CTAs per SM, but with 4096-point lines
// (1024-point sides) a CTA's lines take most of the shared memory
#define TBC_BOUNDS __launch_bounds__(FftE<T>::THREADS, 2)
#define TBC_BOUNDS_LN(LN) __launch_bounds__(FftE<T>::THREADS, (LN) >= 10 ? 1 : 2)
#define TBC_PAIR_BOUNDS(LN) __launch_bounds__(pair_threads<T>(4 << (LN)), (LN) >= 10 ? 1 : 2)

// The pass kernels are instantiated per grid size: LNY = log2 ny (passes A,
// C), LNX = log2 nx (passes B, D).  With the period pad = 4: Px = 4 nx,
// Py = 4 ny.

// ------------------------------------------------------------------ pass A
// grid (ceil(nx / L) row groups, 2 fields, ndir); field 0: cs (E1), 1: sc (E2).
// Per row k1: the mirrored coefficient sequence along x2 (period
// Py) is transformed, multiplied by the transforms of the two parity kernels
// eps_r and transformed back: the linear convolutions give the basis
// transform at j2 = 2t + r of the symmetric box.  Lines: [parity][row].
// The gather of the coefficients is the forward transform's first read, the
// kernel products its last write, and the scatter to Vy the inverse
// transforms' last write: shared memory holds only the transforms.

// coefficient k2 (0 <= k2 < ny) of row k1 for field f, mirrored to the input
// n of a line of length Py
template <typename T, int LNY>
struct GatherA {
  const C<T>* E1;
  const C<T>* E2;
  int row0, nx, f;
  __device__ __forceinline__ C<T> coef(int k1, int k2) const {
    constexpr int ny = 1 << LNY, N = ny - 1;
    C<T> c = czero<T>();
    if (f == 0) {
      if (k2 >= 1) c = E1[k1 * N + (k2 - 1)];
    } else {
      if (k1 >= 1) c = E2[(k1 - 1) * ny + k2];
    }
    return c;
  }
  __device__ __forceinline__ C<T> ld(int l, const C<T>*, int n) const {
    constexpr int ny = 1 << LNY, Py = 4 * ny;
    const int k1 = row0 + l;
    if (k1 >= nx) return czero<T>();
    const bool ycos = f != 0;
    if (n < ny) {
      if (n == 0) return ycos ? cscale<T>(coef(k1, 0), (T)2) : czero<T>();
      return coef(k1, n);
    }
    if (n > Py - ny) {
      const C<T> c = coef(k1, Py - n);
      return ycos ? c : mk<T>(-c.x, -c.y);
    }
    return czero<T>();
  }
};

// last write of the forward transform: the products with the two parity
// kernels, into line l (r = 0) and line L + l (r = 1)
template <typename T, typename G>
struct ParityProducts : G {
  const C<T>* eh;                 // [r][P]
  int P, L, ls;
  C<T>* buf;
  __device__ __forceinline__ void st(int l, C<T>*, int k, C<T> v) const {
    buf[(size_t)l * ls + pidx(k)] = cmul<T>(v, eh[k]);
    buf[(size_t)(L + l) * ls + pidx(k)] = cmul<T>(v, eh[P + k]);
  }
};

// last write of the inverse transforms of pass A: Vy(k1, j), j = 2t + r mod Py
template <typename T, int LNY>
struct ScatterA : LineId<T> {
  C<T>* Vy;                       // this field's [nx][Py] block
  int row0, nx, L;
  __device__ __forceinline__ void st(int lr, C<T>*, int k, C<T> v) const {
    constexpr int Py = 4 << LNY;
    const int r = lr >= L ? 1 : 0, l = lr - r * L;
    const int k1 = row0 + l;
    const int t = k < Py / 2 ? k : k - Py;
    if (k1 >= nx || t < -Py / 4 || t >= Py / 4) return;
    const int j2 = 2 * t + r;
    Vy[(size_t)k1 * Py + (j2 & (Py - 1))] = (j2 == -Py / 2) ? czero<T>() : v;
  }
};

template <typename T, int LNY>
__global__ void TBC_PAIR_BOUNDS(LNY) k_tbcA(const C<T>* __restrict__ x, C<T>* __restrict__ Vy, TbcP p,
                                  const C<T>* __restrict__ tw, const C<T>* __restrict__ eh_c,
                                  const C<T>* __restrict__ eh_s, int lL_) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  C<T>* buf = (C<T>*)sm_raw;
  constexpr int LPY = LNY + 2, Py = 1 << LPY, ls = padded_len(Py);
  const int lL = pairs_per_cta<T>(Py) == 1 ? 0 : lL_, L = 1 << lL;
  const int f = blockIdx.y, d = blockIdx.z;
  const int row0 = blockIdx.x * L;
  ScatterA<T, LNY> sc;
  sc.Vy = Vy + (size_t)(d * 2 + f) * p.nx * Py;
  sc.row0 = row0;
  sc.nx = p.nx;
  sc.L = L;
  ParityProducts<T, GatherA<T, LNY>> fwd;
  fwd.E1 = x + (size_t)d * p.nap;
  fwd.E2 = fwd.E1 + p.n1;
  fwd.row0 = row0;
  fwd.nx = p.nx;
  fwd.f = f;
  fwd.eh = f != 0 ? eh_c : eh_s;
  fwd.P = Py;
  fwd.L = L;
  fwd.ls = ls;
  fwd.buf = buf;
  fft_lines<T, false, LPY, pairs_per_cta<T>(Py), pair_threads<T>(Py)>(buf, ls, L, tw, p.twlog, fwd);
  fft_lines<T, true, LPY, 2 * pairs_per_cta<T>(Py), pair_threads<T>(Py)>(buf, ls, 2 * L, tw, p.twlog, sc);
}

// ------------------------------------------------------------------ pass B
// grid (Py / L column groups, ndir).  Per column j2 and field E1, E2: the
// basis transform along x1 split by the parity of j1 = 2t + r (as in pass A),
// times F(G)(|j1|, |j2|)/(Lx Ly), then the inverse torus transform along x1 at
// the nodes p = 0..nx:  sum_j1 Y(j1) e^{2 pi i j1 p/Px} = Z_0(p) + e^{2 pi i p/Px} Z_1(p),
// Z_r = inverse transform of length Px/2 of Y(2t + r) over t.  The products of
// w are gathered on the way (j2 / Ly times those of E1 minus j1 / Lx times
// those of E2) in two half-length lines, which take the same last transform.
// Fused: the parity products (last write of the forward transform), the
// kernel-table products with the move of t to slot t mod Px/2 (last write of
// the first inverse transforms).  The column gather stays a cooperative pass:
// as a per-line first read it would load one element per 32-byte sector.

// w = s0 g0 - s1 g1, the product with s0 rounded first and the other one fused
// into the difference: said explicitly for FP64, so that the two forms of pass
// B, which take a vector by the size of the batch, give the same bits (the pair
// type's operations are exact about this by themselves).
template <typename T> __device__ __forceinline__ C<T> w_first(C<T> g0, T s0) {
  if constexpr (std::is_same<T, double>::value)
    return make_double2(__dmul_rn(g0.x, s0), __dmul_rn(g0.y, s0));
  else
    return cscale<T>(g0, s0);
}
template <typename T> __device__ __forceinline__ C<T> w_second(C<T> w, C<T> g1, T s1) {
  if constexpr (std::is_same<T, double>::value)
    return make_double2(__fma_rn(-g1.x, s1, w.x), __fma_rn(-g1.y, s1, w.y));
  else
    return csub<T>(w, cscale<T>(g1, s1));
}

// last write of the first inverse transforms of pass B: output t (k = t mod
// Px) of line (r, l), |t| < Px/4, times the kernel table at (|2t + r|, |j2|),
// written to slot t mod Px/2 (other outputs are not needed), and into w
// STAGED: kh holds the rows of the block's columns in shared memory,
// [l][j1 < Px/2]; else kh is the whole quarter box in global memory, [j2][j1]
template <typename T, int LNX, int F, bool STAGED>
struct KhatB : LineId<T> {
  const C<T>* kh;
  C<T>* wl;                       // w: half-length lines [r][l]
  int j0, Py, L;
  T scale;                        // 2 pi / Ly (field 0), 2 pi / Lx (field 1)
  __device__ __forceinline__ void st(int lr, C<T>* line, int k, C<T> v) const {
    constexpr int Px = 4 << LNX, hp = Px / 2, qp = Px / 4;
    int t, u;
    if (k < qp) { t = k; u = k; }
    else if (k >= Px - qp) { t = k - Px; u = k - hp; }
    else return;
    const int r = lr >= L ? 1 : 0, l = lr - r * L;
    const int j = j0 + l;
    const int j1 = 2 * t + r, j2 = j < Py / 2 ? j : j - Py;
    C<T> o = czero<T>();
    if (j1 != -hp && j < Py && j != Py / 2) {
      const int j1a = j1 < 0 ? -j1 : j1;
      if constexpr (STAGED) {
        o = cmul<T>(v, kh[l * hp + j1a]);
      } else {
        const int j2a = j2 < 0 ? -j2 : j2;
        o = cmul<T>(v, kh[(size_t)j2a * hp + j1a]);
      }
    }
    line[pidx(u)] = o;
    C<T>* w = wl + (size_t)lr * padded_len(hp) + pidx(u);
    if (F == 0) *w = w_first<T>(o, (T)j2 * scale);
    else *w = w_second<T>(*w, o, (T)j1 * scale);
  }
};

// pass B stages the two parity kernels and the kernel-table rows of its
// columns in shared memory when lines and tables together take at most
// 100 KB (16-byte types up to 256 points per side); else it
// reads them from global memory (they stay in L2), which leaves room for more
// CTAs per SM: at 512 points per side the pair-of-FP32 pass B of the
// four-layer 512^2 benchmark step went from 16.2 to 9.4 ms (one CTA per SM
// with the staging, two without), and it is the only way at 1024
template <typename T> __host__ __device__ constexpr size_t smem_b_lines(int nx, int lL) {
  return sizeof(C<T>) * ((size_t)2 << lL) * (size_t)(padded_len(4 * nx) + padded_len(2 * nx));
}
template <typename T> __host__ __device__ constexpr size_t smem_b_tables(int nx, int lL) {
  return sizeof(C<T>) * (2 * 4 * (size_t)nx + ((size_t)2 << lL) * nx);
}
template <typename T> __host__ __device__ constexpr bool b_staged(int nx) {
  return smem_b_lines<T>(nx, clog2(pairs_per_cta<T>(4 * nx))) +
             smem_b_tables<T>(nx, clog2(pairs_per_cta<T>(4 * nx))) <= 100 * 1024;
}

// shared memory of pass B: 2L lines, 2L half-length lines of w, then (STAGE)
// the two parity kernels [2][Px] and the kernel-table rows |j2| of the L
// columns [L][Px/2], so that the fused products read shared memory instead of
// waiting on loads
template <typename T, int LNX> struct BShape {
  static constexpr int LPX = LNX + 2, Px = 1 << LPX, nx = 1 << LNX;
  static constexpr int ls = padded_len(Px), lsh = padded_len(Px / 2);
  static constexpr bool STAGE = b_staged<T>(nx);
};

// Z_0 + e^{2 pi i q / Px} Z_1 of the lines at z (stride zs), into W's rows;
// w carries the factor i (TIMES_I)
template <typename T, int LNX, bool TIMES_I>
__device__ __forceinline__ void b_store(const C<T>* z, int zs, C<T>* __restrict__ dst, int j0,
                                        int Py, const C<T>* __restrict__ tw, int sh, int lL) {
  using S = BShape<T, LNX>;
  const int L = 1 << lL;
  for (int idx = threadIdx.x; idx < L * (S::nx + 1); idx += blockDim.x) {
    const int q = idx >> lL, l = idx & (L - 1);
    const int j = j0 + l;
    if (j >= Py) continue;
    const C<T> z0 = z[(size_t)l * zs + pidx(q)];
    const C<T> z1 = z[(size_t)(L + l) * zs + pidx(q)];
    const C<T> o = cadd<T>(z0, cmul<T>(z1, twid<T, true>(tw, q << sh)));
    dst[(size_t)q * Py + j] = TIMES_I ? cmul_i<T>(o) : o;
  }
}

// Field F of pass B.  The field is a template argument: with a loop over the
// two fields the compiler spilled 2-4 KB per thread.
template <typename T, int LNX, int F>
__device__ __forceinline__ void b_field(const C<T>* __restrict__ src, C<T>* __restrict__ dst,
                                     const C<T>* __restrict__ tw, const C<T>* __restrict__ eh,
                                     const C<T>* __restrict__ kh, int j0, int Py,
                                     int twlog, T scale, int lL) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  using S = BShape<T, LNX>;
  constexpr int LPX = S::LPX, Px = S::Px, nx = S::nx, ls = S::ls;
  const int L = 1 << lL;
  C<T>* buf = (C<T>*)sm_raw;
  C<T>* wl = buf + (size_t)2 * L * ls;
  C<T>* eh_sm = wl + (size_t)2 * L * S::lsh;
  const int tid = threadIdx.x, nthr = blockDim.x;
  constexpr bool xcos = F == 0;
  constexpr int ML = 2 * pairs_per_cta<T>(Px), CT = pair_threads<T>(Px);
  if constexpr (S::STAGE) {
    for (int t = tid; t < 2 * Px; t += nthr) eh_sm[t] = eh[t];
  }
  // cooperative, coalesced gather of the L columns (consecutive threads take
  // consecutive columns of a row); the mirrored lines cover every slot but
  // [nx, Px - nx], which is cleared
#pragma unroll 4
  for (int idx = tid; idx < L * nx; idx += nthr) {
    const int k1 = idx >> lL, l = idx & (L - 1);
    const int j = j0 + l;
    const C<T> c = j < Py ? src[(size_t)k1 * Py + j] : czero<T>();
    const C<T> c0 = k1 == 0 ? (xcos ? cscale<T>(c, (T)2) : czero<T>()) : c;
    const C<T> cm = xcos ? c : mk<T>(-c.x, -c.y);
    C<T>* line = buf + (size_t)l * ls;
    line[pidx(k1)] = c0;
    if (k1 > 0) line[pidx(Px - k1)] = cm;
  }
  for (int idx = tid; idx < L * (2 * nx + 1); idx += nthr) {
    const int l = idx / (2 * nx + 1), k = nx + idx - l * (2 * nx + 1);
    buf[(size_t)l * ls + pidx(k)] = czero<T>();
  }
  __syncthreads();
  ParityProducts<T, LineId<T>> fwd;
  fwd.eh = S::STAGE ? eh_sm : eh;
  fwd.P = Px;
  fwd.L = L;
  fwd.ls = ls;
  fwd.buf = buf;
  fft_lines<T, false, LPX, pairs_per_cta<T>(Px), pair_threads<T>(Px)>(buf, ls, L, tw, twlog, fwd);
  KhatB<T, LNX, F, S::STAGE> kb;
  kb.kh = S::STAGE ? eh_sm + 2 * Px : kh;
  kb.wl = wl;
  kb.j0 = j0;
  kb.Py = Py;
  kb.L = L;
  kb.scale = scale;
  fft_lines<T, true, LPX, ML, CT>(buf, ls, 2 * L, tw, twlog, kb);
  fft_lines<T, true, LPX - 1, ML, CT>(buf, ls, 2 * L, tw, twlog);
  b_store<T, LNX, false>(buf, ls, dst, j0, Py, tw, twlog - LPX, lL);
  __syncthreads();
}

template <typename T, int LNX>
__global__ void TBC_PAIR_BOUNDS(LNX) k_tbcB(const C<T>* __restrict__ Vy, C<T>* __restrict__ W, TbcP p,
                                  const C<T>* __restrict__ tw, const C<T>* __restrict__ eh_c,
                                  const C<T>* __restrict__ eh_s, const C<T>* __restrict__ kh,
                                  T ax, T ay, int lL_) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  using S = BShape<T, LNX>;
  constexpr int LPX = S::LPX, Px = S::Px, nx = S::nx;
  const int lL = pairs_per_cta<T>(Px) == 1 ? 0 : lL_, L = 1 << lL;
  C<T>* wl = (C<T>*)sm_raw + (size_t)2 * L * S::ls;
  const int Py = p.Py, d = blockIdx.y, j0 = blockIdx.x * L;
  if constexpr (S::STAGE) {
    C<T>* kh_sm = wl + (size_t)2 * L * S::lsh + 2 * Px;
    for (int idx = threadIdx.x; idx < L * (Px / 2); idx += blockDim.x) {
      const int l = idx >> (LPX - 1), j1 = idx & (Px / 2 - 1);
      const int j = j0 + l;
      const int j2a = j < Py / 2 ? j : Py - j;
      kh_sm[idx] = (j < Py && j != Py / 2) ? kh[(size_t)j2a * (Px / 2) + j1] : czero<T>();
    }
  }
  const C<T>* src = Vy + (size_t)d * 2 * nx * Py;
  const size_t fs = (size_t)(nx + 1) * Py;
  C<T>* dst = W + (size_t)d * 3 * fs;
  b_field<T, LNX, 0>(src, dst, tw, eh_c, kh, j0, Py, p.twlog, ay, lL);
  b_field<T, LNX, 1>(src + (size_t)nx * Py, dst + fs, tw, eh_s, kh, j0, Py, p.twlog, ax, lL);
  fft_lines<T, true, LPX - 1, 2 * pairs_per_cta<T>(Px), pair_threads<T>(Px)>(wl, S::lsh, 2 * L, tw, p.twlog);
  b_store<T, LNX, true>(wl, S::lsh, dst + 2 * fs, j0, Py, tw, p.twlog - LPX, lL);
}

// Pass B for small launches (fewer columns than keep the machine busy): one
// column per CTA with both fields' lines, and those of w, side by side, so a
// CTA goes through three transforms instead of seven.  Lines (stride ls):
// (field f, parity r) at 2 f + r, w at 4 + r.  One FP64 vector at 32 x 32:
// 62 us with k_tbcB, 28 us.
template <typename T, int LNX>
struct ProdsB1 : LineId<T> {     // parity products of both fields' spectra
  const C<T>* eh_c;
  const C<T>* eh_s;
  __device__ __forceinline__ void st(int f, C<T>* line, int k, C<T> v) const {
    constexpr int Px = 4 << LNX, ls = padded_len(Px);
    const C<T>* eh = f == 0 ? eh_c : eh_s;
    line[pidx(k)] = cmul<T>(v, eh[k]);
    line[ls + pidx(k)] = cmul<T>(v, eh[Px + k]);
  }
};
template <typename T, int LNX>
struct KhatB1 : LineId<T> {      // table products; the result stays in slot t mod Px/2
  const C<T>* kh;                // row |j2|
  bool dead;
  __device__ __forceinline__ void st(int lr, C<T>* line, int k, C<T> v) const {
    constexpr int Px = 4 << LNX, hp = Px / 2, qp = Px / 4;
    int t, u;
    if (k < qp) { t = k; u = k; }
    else if (k >= Px - qp) { t = k - Px; u = k - hp; }
    else return;
    const int j1 = 2 * t + (lr & 1);
    line[pidx(u)] = (j1 == -hp || dead) ? czero<T>() : cmul<T>(v, kh[j1 < 0 ? -j1 : j1]);
  }
};
template <typename T, int LNX>
__global__ void TBC_BOUNDS k_tbcB1(const C<T>* __restrict__ Vy, C<T>* __restrict__ W, TbcP p,
                                   const C<T>* __restrict__ tw, const C<T>* __restrict__ eh_c,
                                   const C<T>* __restrict__ eh_s, const C<T>* __restrict__ kh,
                                   T ax, T ay) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  C<T>* buf = (C<T>*)sm_raw;
  using S = BShape<T, LNX>;
  constexpr int LPX = S::LPX, Px = S::Px, nx = S::nx, ls = S::ls;
  const int Py = p.Py, d = blockIdx.y, j = blockIdx.x, tid = threadIdx.x, nthr = blockDim.x;
  const int j2 = j < Py / 2 ? j : j - Py;
  const bool dead = j == Py / 2;
  for (int idx = tid; idx < 2 * Px; idx += nthr) {
    const int f = idx / Px, k = idx % Px;
    const int k1 = k < nx ? k : Px - k;     // mirrored
    C<T> c = czero<T>();
    if (k1 < nx && (f == 0 || k1 > 0)) c = Vy[((size_t)(d * 2 + f) * nx + k1) * Py + j];
    if (k == 0) c = cscale<T>(c, (T)2);
    if (f == 1 && k > nx) c = mk<T>(-c.x, -c.y);
    buf[(size_t)(2 * f) * ls + pidx(k)] = c;
  }
  __syncthreads();
  ProdsB1<T, LNX> fwd;
  fwd.eh_c = eh_c;
  fwd.eh_s = eh_s;
  fft_lines<T, false, LPX, 2>(buf, 2 * ls, 2, tw, p.twlog, fwd);
  KhatB1<T, LNX> kb;
  kb.kh = kh + (size_t)(dead ? 0 : (j2 < 0 ? -j2 : j2)) * (Px / 2);
  kb.dead = dead;
  fft_lines<T, true, LPX, 4>(buf, ls, 4, tw, p.twlog, kb);
  for (int idx = tid; idx < Px; idx += nthr) {
    const int r = idx / (Px / 2), u = idx % (Px / 2);
    const int j1 = 2 * (u < nx ? u : u - Px / 2) + r;
    const C<T> g0 = buf[(size_t)r * ls + pidx(u)], g1 = buf[(size_t)(2 + r) * ls + pidx(u)];
    buf[(size_t)(4 + r) * ls + pidx(u)] =
        w_second<T>(w_first<T>(g0, (T)j2 * ay), g1, (T)j1 * ax);
  }
  __syncthreads();
  fft_lines<T, true, LPX - 1, 6>(buf, ls, 6, tw, p.twlog);
  for (int idx = tid; idx < 3 * (nx + 1); idx += nthr) {
    const int f = idx / (nx + 1), q = idx % (nx + 1);
    const C<T> z0 = buf[(size_t)(2 * f) * ls + pidx(q)], z1 = buf[(size_t)(2 * f + 1) * ls + pidx(q)];
    const C<T> o = cadd<T>(z0, cmul<T>(z1, twid<T, true>(tw, q << (p.twlog - LPX))));
    W[((size_t)(d * 3 + f) * (nx + 1) + q) * Py + j] = f == 2 ? cmul_i<T>(o) : o;
  }
}
// sizes it is built for, and launches small enough for it
__host__ __device__ constexpr bool b1_ok(int ln) { return ln <= 7; }
inline bool b1_use(int Py, int ndir) { return (long long)Py * ndir <= 4LL * sm_count(); }

// ------------------------------------------------------------------ pass C
// grid (ceil((nx+1)/L) row groups, 3 fields, ndir).  Per node row p: inverse
// torus transform along x2 at q = 0..ny, then the trapezoid projection onto
// cos/sin(n pi q/ny) as an extended FFT of length 2 ny.  Fused: the row load
// (first read), the even / odd extension of U(q), q <= ny (last write of the
// inverse transform), the weighted store of Z (last write of the projection).

template <typename T, int LNY>
struct RowC {
  const C<T>* src;                // this field's [nx+1][Py] block
  int r0, nx;
  bool ycos;
  __device__ __forceinline__ C<T> ld(int l, const C<T>*, int n) const {
    constexpr int Py = 4 << LNY;
    const int row = r0 + l;
    return row <= nx ? src[(size_t)row * Py + n] : czero<T>();
  }
  __device__ __forceinline__ void st(int, C<T>* line, int k, C<T> v) const {
    constexpr int ny = 1 << LNY, n2 = 2 * ny;
    if (k > ny) return;
    if (!ycos && (k == 0 || k == ny)) {
      line[pidx(k)] = czero<T>();
      return;
    }
    line[pidx(k)] = v;
    if (k > 0 && k < ny) line[pidx(n2 - k)] = ycos ? v : mk<T>(-v.x, -v.y);
  }
};

template <typename T, int LNY>
struct StoreZ : LineId<T> {
  C<T>* Z;                        // this field's [nx+1][ny+1] block
  int r0, nx;
  bool ycos;
  T w;
  __device__ __forceinline__ void st(int l, C<T>*, int k, C<T> v) const {
    constexpr int ny = 1 << LNY;
    const int row = r0 + l;
    if (k > ny || row > nx) return;
    Z[(size_t)row * (ny + 1) + k] = ycos ? cscale<T>(v, w) : cscale<T>(cmul_i<T>(v), w);
  }
};

template <typename T, int LNY>
__global__ void TBC_BOUNDS_LN(LNY) k_tbcC(const C<T>* __restrict__ W, C<T>* __restrict__ Z, TbcP p,
                                  const C<T>* __restrict__ tw, int lL_) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  C<T>* buf = (C<T>*)sm_raw;
  constexpr int LPY = LNY + 2, Py = 1 << LPY, ny = 1 << LNY, ls = padded_len(Py);
  const int L = lines_per_cta<T>(Py) == 1 ? 1 : 1 << lL_;
  const int f = blockIdx.y, d = blockIdx.z;
  const int r0 = blockIdx.x * L;
  const bool ycos = (f != 0);
  RowC<T, LNY> rc;
  rc.src = W + (size_t)(d * 3 + f) * (p.nx + 1) * Py;
  rc.r0 = r0;
  rc.nx = p.nx;
  rc.ycos = ycos;
  fft_lines<T, true, LPY, lines_per_cta<T>(Py)>(buf, ls, L, tw, p.twlog, rc);
  StoreZ<T, LNY> sz;
  sz.Z = Z + (size_t)(d * 3 + f) * (p.nx + 1) * (ny + 1);
  sz.r0 = r0;
  sz.nx = p.nx;
  sz.ycos = ycos;
  sz.w = (T)p.wy;
  fft_lines<T, false, LNY + 1, lines_per_cta<T>(Py)>(buf, ls, L, tw, p.twlog, sz);
}

// ------------------------------------------------------------------ pass D
// grid (ceil((ny+1)/L) column groups, 3 fields, ndir).  Per column n: the
// trapezoid projection along x1 (extended FFT of length 2 nx), with the
// column gather and extension as the first read and the weighted store of O
// as the last write.
template <typename T, int LNX>
struct ColD {
  const C<T>* src;                // this field's [nx+1][ny+1] block
  C<T>* dst;                      // this field's [nx][ny+1] block
  int c0, ny;
  bool xcos;
  T w;
  __device__ __forceinline__ C<T> ld(int l, const C<T>*, int t) const {
    constexpr int nx = 1 << LNX, n2 = 2 * nx;
    const int col = c0 + l;
    if (col > ny) return czero<T>();
    if (t <= nx) {
      if (!xcos && (t == 0 || t == nx)) return czero<T>();
      return src[(size_t)t * (ny + 1) + col];
    }
    const C<T> r = src[(size_t)(n2 - t) * (ny + 1) + col];
    return xcos ? r : mk<T>(-r.x, -r.y);
  }
  __device__ __forceinline__ void st(int l, C<T>*, int m, C<T> v) const {
    constexpr int nx = 1 << LNX;
    const int col = c0 + l;
    if (m >= nx || col > ny) return;
    dst[(size_t)m * (ny + 1) + col] = xcos ? cscale<T>(v, w) : cscale<T>(cmul_i<T>(v), w);
  }
};

template <typename T, int LNX>
__global__ void TBC_BOUNDS_LN(LNX) k_tbcD(const C<T>* __restrict__ Z, C<T>* __restrict__ O, TbcP p,
                                  const C<T>* __restrict__ tw, int lL_) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  C<T>* buf = (C<T>*)sm_raw;
  constexpr int nx = 1 << LNX, n2 = 2 * nx, ls = padded_len(n2);
  const int L = lines_per_cta<T>(n2) == 1 ? 1 : 1 << lL_;
  const int f = blockIdx.y, d = blockIdx.z;
  ColD<T, LNX> cd;
  cd.src = Z + (size_t)(d * 3 + f) * (nx + 1) * (p.ny + 1);
  cd.dst = O + (size_t)(d * 3 + f) * nx * (p.ny + 1);
  cd.c0 = blockIdx.x * L;
  cd.ny = p.ny;
  cd.xcos = (f != 1);
  cd.w = (T)p.wx;
  fft_lines<T, false, LNX + 1, lines_per_cta<T>(n2)>(buf, ls, L, tw, p.twlog, cd);
}

// ------------------------------------------------------------------ combine
// y = local part of (EJ1)/(uT1) + TBC rows, with the TBC sign that makes T
// the exterior admittance z x curl E^s of (EGa2):
//  row 1: (-1+tau1)E1 + (m pi h/a + vs1)E3 + (h/q)(2k^2 U1 - 2(n pi/b) W)
//  row 2: (-1+tau2)E2 + (n pi h/b + vs2)E3 + (h/c)(2k^2 U2 + 2(m pi/a) W)
//  row 3: (m pi h/a)E1 + (n pi h/b)E2 + (-1+tau3)E3
// One thread per mode pair (m, n), m < nx, n < ny, writing the rows of the
// three components that exist for it, 0 for the modes beyond (mm, nn) of a
// truncated expansion (the operator then maps the kept subspace to itself, as
// does the mode-wise preconditioner); nyp: pitch of O's rows; pm: order of y;
// grid (ceil(nx ny / blockDim), ndir).
template <typename T>
__global__ void k_combine(const C<T>* __restrict__ x, const C<T>* __restrict__ O,
                          const C<T>* __restrict__ top, C<T>* __restrict__ y, long long ys, int nyp,
                          TbcP p, int mm, int nn, ParityMap pm) {
  const int d = blockIdx.y;
  const int mn = blockIdx.x * blockDim.x + threadIdx.x;
  if (mn >= p.nx * p.ny) return;
  const int m = mn >> p.lny, n = mn & (p.ny - 1);
  const C<T>* xd = x + (size_t)d * p.nap;
  C<T>* yd = y + (size_t)d * ys;
  const int N = p.N;
  const size_t fs = (size_t)p.nx * nyp;
  const C<T>* Od = O + (size_t)d * 3 * fs;
  const T pa = (T)p.pia, pb = (T)p.pib, h = (T)p.h, ab = (T)p.ab;
  const T k2 = (T)p.k2x2;
  const int i1 = m * N + (n - 1), i2 = p.n1 + (m - 1) * (N + 1) + n;
  const int i3 = p.n1 + p.n2 + (m - 1) * N + (n - 1);
  const bool has1 = n >= 1, has2 = m >= 1, has3 = m >= 1 && n >= 1;
  const bool kept = m <= mm && n <= nn;
  const C<T> e1 = has1 ? xd[i1] : mk<T>(0, 0);
  const C<T> e2 = has2 ? xd[i2] : mk<T>(0, 0);
  const C<T> e3 = has3 ? xd[i3] : mk<T>(0, 0);
  const size_t o = (size_t)m * nyp + n;
  if (has1) {
    C<T> r = cmul<T>(cadd<T>(mk<T>(-1, 0), top[i1]), e1);
    if (has3) r = cadd<T>(r, cmul<T>(cadd<T>(mk<T>(m * pa * h, 0), top[p.nap + i1]), e3));
    const T s = h / (m == 0 ? ab / 2 : ab / 4);
    const C<T> t = csub<T>(cscale<T>(Od[o], k2), cscale<T>(Od[2 * fs + o], 2 * n * pb));
    yd[pm.on ? pm.e1(m, n) : i1] = kept ? cadd<T>(r, cscale<T>(t, s)) : czero<T>();
  }
  if (has2) {
    C<T> r = cmul<T>(cadd<T>(mk<T>(-1, 0), top[i2]), e2);
    if (has3) r = cadd<T>(r, cmul<T>(cadd<T>(mk<T>(n * pb * h, 0), top[p.nap + i2]), e3));
    const T s = h / (n == 0 ? ab / 2 : ab / 4);
    const C<T> t = cadd<T>(cscale<T>(Od[fs + o], k2), cscale<T>(Od[2 * fs + o], 2 * m * pa));
    yd[pm.on ? pm.e2(m, n) : i2] = kept ? cadd<T>(r, cscale<T>(t, s)) : czero<T>();
  }
  if (has3) {
    C<T> r = cscale<T>(e1, m * pa * h);
    r = cadd<T>(r, cscale<T>(e2, n * pb * h));
    r = cadd<T>(r, cmul<T>(cadd<T>(mk<T>(-1, 0), top[i3]), e3));
    yd[pm.on ? pm.e3(m, n) : i3] = kept ? r : czero<T>();
  }
}

// Explicit instantiation (EXT empty) or its declaration (EXT = extern) of the
// four pass kernels of type T at log2 size LN; lets a type's instantiations
// be compiled in several translation units (in parallel) while one unit
// launches them (TBC_B1_KERNEL: sizes of b1_ok).
#define TBC_B1_KERNEL(EXT, T, LN)                                                             \
  EXT template __global__ void k_tbcB1<T, LN>(const C<T>*, C<T>*, TbcP, const C<T>*,          \
                                              const C<T>*, const C<T>*, const C<T>*, T, T);
#define TBC_PASS_KERNELS(EXT, T, LN)                                                          \
  EXT template __global__ void k_tbcA<T, LN>(const C<T>*, C<T>*, TbcP, const C<T>*,           \
                                             const C<T>*, const C<T>*, int);                  \
  EXT template __global__ void k_tbcB<T, LN>(const C<T>*, C<T>*, TbcP, const C<T>*,           \
                                             const C<T>*, const C<T>*, const C<T>*, T, T,     \
                                             int);                                            \
  EXT template __global__ void k_tbcC<T, LN>(const C<T>*, C<T>*, TbcP, const C<T>*, int);     \
  EXT template __global__ void k_tbcD<T, LN>(const C<T>*, C<T>*, TbcP, const C<T>*, int);

template <typename T> struct Tabs;
template <> struct Tabs<double> {
  static const double2* tw(cavity_ctx* c) { return c->tw64; }
  static const double2* ex(cavity_ctx* c, int k) { return c->ehat_x64[k]; }
  static const double2* ey(cavity_ctx* c, int k) { return c->ehat_y64[k]; }
  static const double2* kh(cavity_ctx* c) { return c->khat64; }
  static const double2* top(cavity_ctx* c) { return c->top64; }
};

// shared memory of each pass (bytes) at 2^lL lines (or pairs) per CTA
template <typename T> static size_t smem_a(int ny, int lL) {
  return sizeof(C<T>) * ((size_t)2 << lL) * padded_len(4 * ny);
}
template <typename T> static size_t smem_b(int nx, int lL) {
  return smem_b_lines<T>(nx, lL) + (b_staged<T>(nx) ? smem_b_tables<T>(nx, lL) : 0);
}
template <typename T> static size_t smem_c(int ny, int lL) {
  return sizeof(C<T>) * ((size_t)1 << lL) * padded_len(4 * ny);
}
template <typename T> static size_t smem_d(int nx, int lL) {
  return sizeof(C<T>) * ((size_t)1 << lL) * padded_len(2 * nx);
}

// the last kept mode of each axis
static int last_m(const cavity_ctx* ctx) { return ctx->desc.modes_m > 0 ? ctx->desc.modes_m : ctx->g.M; }
static int last_n(const cavity_ctx* ctx) { return ctx->desc.modes_n > 0 ? ctx->desc.modes_n : ctx->g.N; }

// opt every instantiation of kernel K into the device's shared-memory maximum
// once per process
template <typename K> static cavity_status smem_once(cavity_ctx* ctx, K kern, DeviceFlag& done) {
  if (!done) {
    CK(allow_max_smem(kern));
    done.set();
  }
  return CAVITY_OK;
}

// launch-accounting class of pass `k` (0..4: A, B, C, D, combine) for type T
template <typename T> static int kclass(int k) {
  if (std::is_same<T, double>::value) return KC_TBC_A64 + k;
  return KC_TBC_AP + k;
}

template <typename T>
cavity_status launch_apply(cavity_ctx* ctx, int ndir, const C<T>* x, C<T>* y, void* work,
                           long long ystride, const ParityMap& pm) {
  if (!ctx->g.fft_ok) {
    ctx->err = "the FFT operator needs the convolution period 4 on both axes";
    return CAVITY_EINVAL;
  }
  if (ystride < 0) ystride = ctx->g.nap;
  const Geo& g = ctx->g;
  const int pl = clog2(pairs_per_cta<T>(4 * g.ny)), pb = clog2(pairs_per_cta<T>(4 * g.nx));
  const size_t need = std::max(
      std::max(smem_a<T>(g.ny, pl), smem_b<T>(g.nx, pb)),
      std::max(smem_c<T>(g.ny, clog2(lines_per_cta<T>(4 * g.ny))),
               smem_d<T>(g.nx, clog2(lines_per_cta<T>(2 * g.nx)))));
  if (need > (size_t)smem_optin()) {
    ctx->err = "grid too large for the shared-memory transforms";
    return CAVITY_EINVAL;
  }
  TbcP p = make_params(ctx);
  size_t vy = (size_t)ndir * 2 * g.nx * g.Py;
  size_t z = (size_t)ndir * 3 * (g.nx + 1) * (g.ny + 1);
  C<T>* R1 = (C<T>*)work;                      // Vy, later Z
  C<T>* R2 = R1 + std::max(vy, z);             // W, later O
  cudaStream_t st = ctx->stream;
  const C<T>* tw = Tabs<T>::tw(ctx);
  CKS(dispatch_log<CAV_LOG_MIN, CAV_LOG_MAX>(g.lny, [&](auto c) -> cavity_status {
    constexpr int LN = decltype(c)::value;
    const CtaLines cl = cta_lines(clog2(pairs_per_cta<T>(4 << LN)), 2, fft_tpl<T>(4 << LN),
                                  pair_threads<T>(4 << LN), g.nx,
                                  2LL * ndir);
    static DeviceFlag done;
    CKS(smem_once(ctx, k_tbcA<T, LN>, done));
    KScope ks_(ctx, kclass<T>(0));
    k_tbcA<T, LN><<<dim3(cl.blocks(g.nx), 2, ndir), cl.threads, smem_a<T>(g.ny, cl.lL), st>>>(
        x, R1, p, tw, Tabs<T>::ey(ctx, 0), Tabs<T>::ey(ctx, 1), cl.lL);
    return CAVITY_OK;
  }));
  CKS(dispatch_log<CAV_LOG_MIN, CAV_LOG_MAX>(g.lnx, [&](auto c) -> cavity_status {
    constexpr int LN = decltype(c)::value;
    if constexpr (b1_ok(LN)) {
      if (b1_use(g.Py, ndir)) {
        static DeviceFlag done1;
        CKS(smem_once(ctx, k_tbcB1<T, LN>, done1));
        KScope ks_(ctx, kclass<T>(1));
        k_tbcB1<T, LN><<<dim3(g.Py, ndir), std::max(64, std::min(FftE<T>::THREADS, 6 * fft_tpl<T>(4 << LN))),
                         sizeof(C<T>) * 6 * (size_t)padded_len(4 << LN), st>>>(
            R1, R2, p, tw, Tabs<T>::ex(ctx, 0), Tabs<T>::ex(ctx, 1), Tabs<T>::kh(ctx),
            T(2.0 * M_PI / g.Lx), T(2.0 * M_PI / g.Ly));
        return CAVITY_OK;
      }
    }
    const CtaLines cl = cta_lines(clog2(pairs_per_cta<T>(4 << LN)), 2, fft_tpl<T>(4 << LN),
                                  pair_threads<T>(4 << LN), g.Py,
                                  ndir);
    static DeviceFlag done;
    CKS(smem_once(ctx, k_tbcB<T, LN>, done));
    KScope ks_(ctx, kclass<T>(1));
    k_tbcB<T, LN><<<dim3(cl.blocks(g.Py), ndir), cl.threads, smem_b<T>(g.nx, cl.lL), st>>>(
        R1, R2, p, tw, Tabs<T>::ex(ctx, 0), Tabs<T>::ex(ctx, 1), Tabs<T>::kh(ctx),
        T(2.0 * M_PI / g.Lx), T(2.0 * M_PI / g.Ly), cl.lL);
    return CAVITY_OK;
  }));
  CKS(dispatch_log<CAV_LOG_MIN, CAV_LOG_MAX>(g.lny, [&](auto c) -> cavity_status {
    constexpr int LN = decltype(c)::value;
    const CtaLines cl = cta_lines(clog2(lines_per_cta<T>(4 << LN)), 1, fft_tpl<T>(4 << LN),
                                  FftE<T>::THREADS, g.nx + 1,
                                  3LL * ndir);
    static DeviceFlag done;
    CKS(smem_once(ctx, k_tbcC<T, LN>, done));
    KScope ks_(ctx, kclass<T>(2));
    k_tbcC<T, LN><<<dim3(cl.blocks(g.nx + 1), 3, ndir), cl.threads, smem_c<T>(g.ny, cl.lL), st>>>(
        R2, R1, p, tw, cl.lL);
    return CAVITY_OK;
  }));
  CKS(dispatch_log<CAV_LOG_MIN, CAV_LOG_MAX>(g.lnx, [&](auto c) -> cavity_status {
    constexpr int LN = decltype(c)::value;
    const CtaLines cl = cta_lines(clog2(lines_per_cta<T>(2 << LN)), 1, fft_tpl<T>(2 << LN),
                                  FftE<T>::THREADS, g.ny + 1,
                                  3LL * ndir);
    static DeviceFlag done;
    CKS(smem_once(ctx, k_tbcD<T, LN>, done));
    KScope ks_(ctx, kclass<T>(3));
    k_tbcD<T, LN><<<dim3(cl.blocks(g.ny + 1), 3, ndir), cl.threads, smem_d<T>(g.nx, cl.lL), st>>>(
        R1, R2, p, tw, cl.lL);
    return CAVITY_OK;
  }));
  {
    KScope ks_(ctx, kclass<T>(4));
    const int eb = elem_block((long long)g.nx * g.ny * ndir);
    k_combine<T><<<dim3((g.nx * g.ny + eb - 1) / eb, ndir), eb, 0, st>>>(x, R2, Tabs<T>::top(ctx), y,
                                                                         ystride, g.ny + 1, p,
                                                                         last_m(ctx), last_n(ctx), pm);
  }
  CK(cudaGetLastError());
  return CAVITY_OK;
}
