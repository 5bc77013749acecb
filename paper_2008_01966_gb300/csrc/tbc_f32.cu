// The FP32 aperture operator (inner iterations of the mixed-precision solve):
// the passes of tbc_apply.cuh with register-resident group transforms
// (gfft.cuh).
//
// What differs from the generic passes:
//  * Two basis transforms instead of three.  E1 is a sine series in x2 and E2
//    one in x1, so both vanish on the edges they are differentiated across and
//    the third field w = d2 E1 - d1 E2 has, exactly, the transform
//      F(w)(xi) = 2 pi i (xi2 F(E1)(xi) - xi1 F(E2)(xi)).
//    Pass A transforms E1 and E2 only, and pass B forms F(w) pointwise between
//    its first inverse transforms and the products with F(G).
//  * Pass B chains forward transform, kernel product, inverse transform,
//    table product and second inverse transform in registers; shared memory
//    holds only the transposes.  Two groups of lanes work on a column, one per
//    field; the third field's two half-length transforms go one to each.
//  * The intermediate grids are stored for the reader: Vy as [j2][k1] and U as
//    [j2][p], so pass B reads and writes whole lines; passes A and C turn
//    several rows at once through shared memory (32-byte pieces).
// Bound: instruction issue (pass B at 256 x 256, 16 vectors: issue slots 65 %
// busy, shared-memory and L1 pipe 64 %, 122 MB of DRAM traffic in 0.25 ms), three
// blocks of 128 threads per SM.  Measured on a GB300, us per launch of pass B,
// against lines kept in shared memory with three basis transforms (every
// column's forward transform done twice):
//   64 x 64, 64 vectors 147 -> 56;  256 x 256, 64 vectors 2624 -> 964;
//   512 x 256, 5 vectors 496 -> 221;  512 x 512, 8 vectors 1554 -> 831;
//   1024 x 1024, 3 vectors 2981 -> 1435.
// Sides of 4 and 8 (lines of 16 and 32 points, 32 of them in a block of pass A),
// us per operator, the generic passes and these: 256 x 4, 8 vectors 76 -> 54;
// 512 x 8, 8 vectors 80 -> 63; 8 x 8, one vector 51 -> 49.
// The three passes around it (A, C, D), 256 x 256, 64 vectors: 670 -> 410.
// Error against 64 bits (relative, random vectors, 16 .. 1024 per side):
// 0.9e-7 .. 2.1e-7, before 1.0e-7 .. 3.1e-7; on right-hand sides and solutions
// (smooth vectors) within +-15 % of before up to 512, smaller at 1024.
#include "gfft.cuh"
#include "tbc_apply.cuh"

// ------------------------------------------------------------------ lane tables
__global__ void k_lane_tab(float2* __restrict__ out, int n, int LG, int RV) {
  const int size = lane_tab_size(n, LG);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= size) return;
  int num, den;   // exp(-2 pi i num / den)
  const int h0 = lane_tab_half(n, LG), p0 = lane_tab_post(n, LG);
  if (i < n) {
    num = (i / LG) * (i % LG);
    den = n;
  } else if (i < h0) {
    num = ((i - n) / RV) * ((i - n) % RV);
    den = LG;
  } else if (i < h0 + n / 2) {
    const int k = i - h0;
    num = (k / LG) * (k % LG);
    den = n / 2;
  } else if (i < p0) {
    const int k = i - h0 - n / 2, rv = RV / 2;
    num = (k / rv) * (k % rv);
    den = LG;
  } else {
    num = -(i - p0);
    den = n;
  }
  double s, c;
  sincospi(-2.0 * (double)(num % den) / (double)den, &s, &c);
  out[i] = make_float2((float)c, (float)s);
}

cavity_status launch_lane_tables(cavity_ctx* ctx) {
  const Geo& g = ctx->g;
  for (int ax = 0; ax < 2; ++ax) {
    const int ln = ax == 0 ? g.lnx : g.lny, n = 4 << ln;
    CKS(dispatch_log<CAV_LOG_MIN, CAV_LOG_MAX>(ln, [&](auto c) -> cavity_status {
      constexpr int LN = decltype(c)::value;
      using S = GShape<LN + 2>;
      const int sz = lane_tab_size(n, S::LG);
      CK(cudaMalloc(&ctx->lane_tab[ax], sizeof(float2) * sz));
      KScope ks_(ctx, KC_SETUP);
      k_lane_tab<<<(sz + 255) / 256, 256, 0, ctx->stream>>>(ctx->lane_tab[ax], n, S::LG, S::RV);
      // the field's lines, of 2 << ln points
      if constexpr (LN >= FIELD_F32_LOG_MIN) {
        using SF = GShape<LN + 1>;
        const int szf = lane_tab_size(n / 2, SF::LG);
        CK(cudaMalloc(&ctx->lane_tab_f[ax], sizeof(float2) * szf));
        k_lane_tab<<<(szf + 255) / 256, 256, 0, ctx->stream>>>(ctx->lane_tab_f[ax], n / 2, SF::LG,
                                                              SF::RV);
      }
      return CAVITY_OK;
    }));
  }
  CK(cudaGetLastError());
  return CAVITY_OK;
}

// ------------------------------------------------------------------ shapes
// LN = log2 of the axis' intervals; lines of n = 4 << LN points.  Blocks have
// at least 128 threads; with 32 values (64 registers) of the line and as many
// of its spectrum per lane, three blocks of 128 run on an SM.
// Pitch of a line of U (nx + 1 nodes): 32-byte aligned, but packed on sides of 4
// and 8, so that Vt and U fit what the generic passes' Vy and W take
// (apply_work_bytes), in units of Py: 2 nx + 3 (nx + 4) <= 6 nx + 3 from nx = 9.
__host__ __device__ constexpr int u_pitch(int nx) { return nx >= 16 ? nx + 4 : nx + 1; }
template <int LN> struct F32Shape {
  using S = GShape<LN + 2>;
  static constexpr int N = 4 << LN, LG = S::LG, RV = S::RV, H = RV / 2, Q4 = RV / 4;
  static constexpr int NT = 2 * LG > 128 ? 2 * LG : 128;
  static constexpr int TILE = GTile<LG, RV>::SIZE;
  static constexpr int R = NT / LG;        // rows per block of pass A
  static constexpr int CB = NT / (2 * LG); // columns per block of pass B
  static constexpr int CPITCH = u_pitch(1 << LN);
};
#define F32_BOUNDS(LN) __launch_bounds__(F32Shape<LN>::NT, (LN) >= 10 ? 1 : 3)

// ------------------------------------------------------------------ pass A
// grid (ceil(nx / R) row groups, 2 fields, ndir); field 0: E1 (sine in x2), 1: E2
// (cosine).  Group g of the block transforms row k1 = R blockIdx.x + g; both
// parities' results are collected in shared memory and written to
// Vt[d][f][j2][k1], R rows (consecutive k1) at a time.
template <int LN> struct SmemA {
  using F = F32Shape<LN>;
  // row pitch of the collected results: half-warps reading R rows x 16/R
  // columns hit distinct banks
  static constexpr int OP = F::N / 2 + (F::R >= 16 ? 1 : 16 / F::R);
  static constexpr size_t BYTES = sizeof(float2) * (F::R * F::TILE + 2 * F::R * OP);
};
// (At 512 and 128 intervals three blocks per SM would spill 160-440 bytes per
// thread: 512 x 512, 8 vectors, 193 us with three, 162 us with two.)
// PART: fewer rows than a block takes (nx < R); the guards of this case cost 4 %
// of the pass at 256 x 256 and 16 vectors.
template <int LNY, bool PART>
__global__ void __launch_bounds__(F32Shape<LNY>::NT, LNY >= 10 ? 1 : (LNY == 9 || LNY == 7) ? 2 : 3)
    k_opA(const float2* __restrict__ x, float2* __restrict__ Vt, TbcP p,
          const float2* __restrict__ lt, const float2* __restrict__ eh_c,
          const float2* __restrict__ eh_s) {
  using F = F32Shape<LNY>;
  constexpr int LG = F::LG, RV = F::RV, Q4 = F::Q4, n = F::N, ny = 1 << LNY, NN = ny - 1;
  constexpr int R = F::R, OP = SmemA<LNY>::OP;
  extern __shared__ __align__(16) float2 sm2[];
  const int f = blockIdx.y, d = blockIdx.z;
  const int g = threadIdx.x / LG, l = threadIdx.x % LG;
  const int k1 = blockIdx.x * R + g;
  float2* tile = sm2 + g * F::TILE;
  float2* outs = sm2 + R * F::TILE;
  const float2* E1 = x + (size_t)d * p.nap;
  const float2* src = f == 0 ? E1 + (size_t)k1 * NN - 1 : E1 + p.n1 + (size_t)(k1 - 1) * ny;
  const bool has = (!PART || k1 < p.nx) && (f == 0 || k1 >= 1);
  float2 v[RV];
#pragma unroll
  for (int r = 0; r < Q4; ++r) {
    const int k2 = l + LG * r;
    float2 c = (has && (f == 1 || k2 >= 1)) ? src[k2] : make_float2(0.f, 0.f);
    if (k2 == 0) c = make_float2(2.f * c.x, 2.f * c.y);
    v[r] = c;
    const int km = LG * (Q4 - r) - l;   // the mirrored slot RV - Q4 + r: 1 .. ny
    c = (has && km < ny) ? src[km] : make_float2(0.f, 0.f);
    v[RV - Q4 + r] = f == 1 ? c : make_float2(-c.x, -c.y);
  }
  gfft<false, LG, RV, true>(v, tile, l, lt, 1 + g);
  float2 z[RV];
#pragma unroll
  for (int i = 0; i < RV; ++i) z[i] = v[i];
  const float2* eh = f != 0 ? eh_c : eh_s;
#pragma unroll 1
  for (int r = 0; r < 2; ++r) {
#pragma unroll
    for (int i = 0; i < RV; ++i) v[i] = cmul<float>(z[i], __ldg(eh + r * n + l + LG * i));
    gfft<true, LG, RV>(v, tile, l, lt, 1 + g);
    float2* o = outs + (size_t)(r * R + g) * OP;
#pragma unroll
    for (int s = 0; s < F::H; ++s) {
      // slot u = t mod n/2, t = l + LG s or that minus n/2; t = -n/4, r = 0 is
      // the Nyquist line
      float2 w = s < Q4 ? v[s] : v[s + F::H];
      if (s == Q4 && l == 0 && r == 0) w = make_float2(0.f, 0.f);
      o[l + LG * s] = w;
    }
  }
  __syncthreads();
  float2* dst = Vt + (size_t)(d * 2 + f) * n * p.nx + blockIdx.x * R;
  for (int i = threadIdx.x; i < n * R; i += F::NT) {
    const int row = i % R, c = i / R, r = c / (n / 2), u = c % (n / 2);
    const int t = u < n / 4 ? u : u - n / 2;
    if (!PART || blockIdx.x * R + row < p.nx)
      dst[(size_t)((2 * t + r) & (n - 1)) * p.nx + row] = outs[(r * R + row) * OP + u];
  }
}

// ------------------------------------------------------------------ pass B
// grid (Py / CB column groups, ndir).  LG <= 32: warp w of the block works on
// field w & 1 of the columns of pair w >> 1 (32 / LG columns); LG > 32: the
// first LG threads on field 0, the others on field 1.
template <int LN> struct SmemB {
  using F = F32Shape<LN>;
  // per column: two tiles, the exchange line, three fields' r = 0 results
  static constexpr int COL = 2 * F::TILE + F::N / 2 + 3 * F::CPITCH;
  static constexpr size_t BYTES = sizeof(float2) * F::CB * COL;
};
template <int LNX>
__global__ void F32_BOUNDS(LNX)
    k_opB(const float2* __restrict__ Vt, float2* __restrict__ Ut, TbcP p,
          const float2* __restrict__ lt, const float2* __restrict__ eh_c,
          const float2* __restrict__ eh_s, const float2* __restrict__ kh, float ax, float ay) {
  using F = F32Shape<LNX>;
  constexpr int LG = F::LG, RV = F::RV, Q4 = F::Q4, H = F::H, n = F::N, nx = 1 << LNX;
  constexpr int CP = F::CPITCH, CB = F::CB;
  extern __shared__ __align__(16) float2 sm2[];
  const int d = blockIdx.y, tid = threadIdx.x;
  int f, col, bar, pbar = 0;
  const int l = tid % LG;
  if constexpr (LG <= 32) {
    const int w = tid >> 5;
    f = w & 1;
    pbar = 1 + (w >> 1);
    col = (w >> 1) * (32 / LG) + (tid & 31) / LG;
    bar = 0;
  } else {
    f = tid / LG;
    col = 0;
    bar = 1 + f;
  }
  auto pair_wait = [&]() {
    if constexpr (F::NT == 64 || 2 * LG == F::NT) __syncthreads();
    else asm volatile("bar.sync %0, 64;" ::"r"(pbar) : "memory");
  };
  // columns of the block: tiles of field 0, tiles of field 1, exchange, results
  float2* tile = sm2 + (f * CB + col) * F::TILE;
  float2* xch = sm2 + 2 * CB * F::TILE + col * (n / 2);
  float2* res = sm2 + 2 * CB * F::TILE + CB * (n / 2) + col * 3 * CP;
  const int Py = p.Py, hy = Py / 2;
  const int j = blockIdx.x * CB + col;
  const int js = j < hy ? j : j - Py;          // signed frequency
  const bool dead = j == hy;                   // the Nyquist line
  const int j2a = dead ? 0 : (js < 0 ? -js : js);
  const float2* src = Vt + ((size_t)(d * 2 + f) * Py + j) * nx;
  float2 v[RV];
#pragma unroll
  for (int r = 0; r < Q4; ++r) {
    const int k = l + LG * r;
    float2 c = src[k];
    if (k == 0) c = f == 0 ? make_float2(2.f * c.x, 2.f * c.y) : make_float2(0.f, 0.f);
    v[r] = c;
    const int km = LG * (Q4 - r) - l;          // 1 .. nx
    c = km < nx ? src[km] : make_float2(0.f, 0.f);
    v[RV - Q4 + r] = f == 0 ? c : make_float2(-c.x, -c.y);
  }
  gfft<false, LG, RV, true>(v, tile, l, lt, bar);
  float2 z[RV];
#pragma unroll
  for (int i = 0; i < RV; ++i) z[i] = v[i];
  const float2* eh = f == 0 ? eh_c : eh_s;
  const float2* lth = lt + lane_tab_half(n, LG);
  const float2* post = lt + lane_tab_post(n, LG);
  const float wy = ay * (float)js;
  float2* dst = Ut + ((size_t)d * 3 * Py + j) * CP;
  const size_t fs = (size_t)Py * CP;
#pragma unroll 1
  for (int r = 0; r < 2; ++r) {
#pragma unroll
    for (int i = 0; i < RV; ++i) v[i] = cmul<float>(z[i], __ldg(eh + r * n + l + LG * i));
    gfft<true, LG, RV>(v, tile, l, lt, bar);
    // times F(G)/(Lx Ly) at j1 = 2t + r, kept in slot t mod n/2; the table is
    // stored by the parity of |j1| (kh[j2][parity][|j1| / 2])
    float2 q[H];
    const float2* kr = kh + ((size_t)j2a * 2 + r) * nx;
#pragma unroll
    for (int s = 0; s < H; ++s) {
      const int u = l + LG * s;
      const int ki = s < Q4 ? u : n / 2 - u - r;
      float2 kv = make_float2(0.f, 0.f);
      if (ki < nx && !dead) kv = __ldg(kr + ki);   // ki = nx: t = -n/4, the Nyquist line
      q[s] = cmul<float>(s < Q4 ? v[s] : v[s + H], kv);
    }
    if (f != r) {
#pragma unroll
      for (int s = 0; s < H; ++s) xch[l + LG * s] = q[s];
    }
    pair_wait();
    auto finish = [&](int fo, float2(&c)[H]) {
      // nodes p = l + LG s, and p = nx (s = Q4, l = 0)
#pragma unroll
      for (int s = 0; s <= Q4; ++s) {
        const int pn = l + LG * s;
        if (s == Q4 && l != 0) break;
        if (r == 0) {
          res[fo * CP + pn] = c[s];
        } else {
          const float2 o = cadd<float>(res[fo * CP + pn], cmul<float>(c[s], __ldg(post + pn)));
          // w carries the factor i
          dst[fo * fs + pn] = fo == 2 ? make_float2(-o.y, o.x) : o;
        }
      }
    };
    if (f == r) {
      float2 w[H];
#pragma unroll
      for (int s = 0; s < H; ++s) {
        const int u = l + LG * s, t = s < Q4 ? u : u - n / 2;
        const float2 o = xch[u];
        const float2 g0 = f == 0 ? q[s] : o, g1 = f == 0 ? o : q[s];
        const float wx = ax * (float)(2 * t + r);
        w[s] = make_float2(wy * g0.x - wx * g1.x, wy * g0.y - wx * g1.y);
      }
      gfft<true, LG, H>(w, tile, l, lth, bar);
      finish(2, w);
    }
    gfft<true, LG, H>(q, tile, l, lth, bar);
    finish(f, q);
  }
}

// ------------------------------------------------------------------ pass C
// grid (ceil((nx + 1) / R) node-row groups, 3 fields, ndir): row p of the
// torus grid, its inverse transform along x2 at the nodes q = 0..ny, and the
// trapezoid projection onto cos/sin(n pi q / ny), n < ny, as a transform of the
// even or odd extension (length 2 ny).  The R rows are gathered from
// U[j2][p] through shared memory (PACKED: of the pitch of sides of 4 and 8; a
// pitch by size or as an argument cost 1 - 3 % of the pass at 256 x 256).
template <int LN> struct SmemC {
  using F = F32Shape<LN>;
  static constexpr int NT = F::LG == 64 ? 256 : F::NT;
  static constexpr int R = NT / F::LG;
  // a row's line, later its tile; the pitch keeps the gather's writes (R rows
  // of one column) on distinct banks
  static constexpr int LP = (F::TILE > F::N ? F::TILE : F::N) / 16 * 16 + 16 + (R >= 16 ? 1 : 16 / R);
  static constexpr size_t BYTES = sizeof(float2) * R * LP;
};
template <int LNY, bool PACKED>
__global__ void __launch_bounds__(SmemC<LNY>::NT, LNY >= 10 ? 2 : (SmemC<LNY>::NT == 256 ? 2 : 4))
    k_opC(const float2* __restrict__ Ut, float2* __restrict__ Z, TbcP p,
          const float2* __restrict__ lt) {
  using F = F32Shape<LNY>;
  constexpr int LG = F::LG, RV = F::RV, Q4 = F::Q4, H = F::H, n = F::N, ny = 1 << LNY;
  constexpr int R = SmemC<LNY>::R, LP = SmemC<LNY>::LP, NT = SmemC<LNY>::NT;
  extern __shared__ __align__(16) float2 sm2[];
  const int f = blockIdx.y, d = blockIdx.z;
  const int g = threadIdx.x / LG, l = threadIdx.x % LG;
  const int p0 = blockIdx.x * R, cp = p.nx + 1, up = p.nx + (PACKED ? 1 : 4);   // u_pitch
  const float2* src = Ut + (size_t)(d * 3 + f) * n * up + p0;
#pragma unroll 16
  for (int i = threadIdx.x; i < n * R; i += NT) {
    const int row = i % R, j = i / R;
    sm2[row * LP + j] = p0 + row < cp ? src[(size_t)j * up + row] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  float2* line = sm2 + g * LP;
  float2 v[RV];
#pragma unroll
  for (int r = 0; r < RV; ++r) v[r] = line[l + LG * r];
  group_sync<LG>(1 + g);
  gfft<true, LG, RV>(v, line, l, lt, 1 + g);
  const bool ycos = f != 0;
  float2 u[H];
#pragma unroll
  for (int s = 0; s < Q4; ++s) {
    u[s] = v[s];
    if (s == 0 && l == 0 && !ycos) u[s] = make_float2(0.f, 0.f);
    line[l + LG * s] = u[s];
  }
  if (l == 0) line[ny] = ycos ? v[Q4] : make_float2(0.f, 0.f);
  group_sync<LG>(1 + g);
#pragma unroll
  for (int s = Q4; s < H; ++s) {
    const float2 m = line[2 * ny - (l + LG * s)];
    u[s] = ycos || (s == Q4 && l == 0) ? m : make_float2(-m.x, -m.y);
  }
  group_sync<LG>(1 + g);
  gfft<false, LG, H>(u, line, l, lt + lane_tab_half(n, LG), 1 + g);
  if (p0 + g >= cp) return;
  float2* dst = Z + ((size_t)(d * 3 + f) * cp + p0 + g) * ny;
  const float w = (float)p.wy;
#pragma unroll
  for (int s = 0; s < Q4; ++s)
    dst[l + LG * s] = ycos ? make_float2(w * u[s].x, w * u[s].y)
                           : make_float2(-w * u[s].y, w * u[s].x);
}

// ------------------------------------------------------------------ pass D
// grid (ny / R column groups, 3 fields, ndir): column n of Z[p][n], its
// trapezoid projection along x1 (length 2 nx), into O[m][n], m < nx.
template <int LN> struct SmemD {
  using F = F32Shape<LN>;
  static constexpr int NT = F::NT;
  static constexpr int R = NT / F::LG;
  static constexpr int HT = GTile<F::LG, F::H>::SIZE;   // tile of the half-length transform
  static constexpr int LN1 = (1 << LN) + 1;
  static constexpr int LP = (HT > LN1 ? HT : LN1) / 16 * 16 + 16 + (R >= 16 ? 1 : 16 / R);
  static constexpr size_t BYTES = sizeof(float2) * R * LP;
};
template <int LNX>
__global__ void __launch_bounds__(SmemD<LNX>::NT, LNX >= 10 ? 2 : 5)
    k_opD(const float2* __restrict__ Z, float2* __restrict__ O, TbcP p,
          const float2* __restrict__ lt) {
  using F = F32Shape<LNX>;
  constexpr int LG = F::LG, Q4 = F::Q4, H = F::H, n = F::N, nx = 1 << LNX;
  constexpr int R = SmemD<LNX>::R, LP = SmemD<LNX>::LP, NT = SmemD<LNX>::NT;
  extern __shared__ __align__(16) float2 sm2[];
  const int f = blockIdx.y, d = blockIdx.z, ny = p.ny;
  const int g = threadIdx.x / LG, l = threadIdx.x % LG;
  const int c0 = blockIdx.x * R;
  const float2* src = Z + (size_t)(d * 3 + f) * (nx + 1) * ny + c0;
  // ny may be smaller than R: the missing columns are zero and not written
#pragma unroll 8
  for (int i = threadIdx.x; i < (nx + 1) * R; i += NT) {
    const int col = i % R, q = i / R;
    sm2[col * LP + q] = c0 + col < ny ? src[(size_t)q * ny + col] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  float2* line = sm2 + g * LP;
  const bool xcos = f != 1;
  float2 u[H];
#pragma unroll
  for (int s = 0; s < H; ++s) {
    const int t = l + LG * s;
    float2 m = line[t <= nx ? t : 2 * nx - t];
    if (!xcos) {
      if (t == 0 || t == nx) m = make_float2(0.f, 0.f);
      else if (t > nx) m = make_float2(-m.x, -m.y);
    }
    u[s] = m;
  }
  group_sync<LG>(1 + g);
  gfft<false, LG, H>(u, line, l, lt + lane_tab_half(n, LG), 1 + g);
  const float w = (float)p.wx;
#pragma unroll
  for (int s = 0; s < Q4; ++s)
    line[l + LG * s] = xcos ? make_float2(w * u[s].x, w * u[s].y)
                            : make_float2(-w * u[s].y, w * u[s].x);
  __syncthreads();
  float2* dst = O + (size_t)(d * 3 + f) * nx * ny + c0;
  for (int i = threadIdx.x; i < nx * R; i += NT) {
    const int col = i % R, m = i / R;
    if (c0 + col < ny) dst[(size_t)m * ny + col] = sm2[col * LP + m];
  }
}

// ------------------------------------------------------------------ launch
// kernel table by parity of j1: kh[j2][parity][j1 / 2]
__global__ void k_khat_split(const float2* __restrict__ in, float2* __restrict__ out, int hx, int hy) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= (long long)hx * hy) return;
  const int j2 = (int)(i / hx), j1 = (int)(i - (long long)j2 * hx);
  out[(size_t)j2 * hx + (j1 & 1) * (hx / 2) + (j1 >> 1)] = in[i];
}
cavity_status launch_khat_split(cavity_ctx* ctx) {
  const Geo& g = ctx->g;
  const size_t n = (size_t)(g.Px / 2) * (g.Py / 2);
  CK(table_alloc(&ctx->khat32s, n));
  KScope ks_(ctx, KC_SETUP);
  k_khat_split<<<(unsigned)((n + 255) / 256), 256, 0, ctx->stream>>>(ctx->khat32, ctx->khat32s,
                                                                    g.Px / 2, g.Py / 2);
  CK(cudaGetLastError());
  return CAVITY_OK;
}

// y = A x in FP32, on every grid of the FFT operator (the options that used to
// choose a pass by its transform are accepted and choose nothing)
template <>
cavity_status launch_apply<float>(cavity_ctx* ctx, int ndir, const float2* x, float2* y,
                                  void* work, long long ystride, const ParityMap& pm) {
  const Geo& g = ctx->g;
  if (!g.fft_ok) {
    ctx->err = "the FFT operator needs the convolution period 4 on both axes";
    return CAVITY_EINVAL;
  }
  if (ystride < 0) ystride = g.nap;
  TbcP p = make_params(ctx);
  cudaStream_t st = ctx->stream;
  // Vt and Z share one region, U and O the other (u_pitch: they fit)
  const size_t vt = (size_t)ndir * 2 * g.nx * g.Py, z = (size_t)ndir * 3 * (g.nx + 1) * g.ny;
  float2* R1 = (float2*)work;
  float2* R2 = R1 + std::max(vt, z);
  CKS(dispatch_log<CAV_LOG_MIN, CAV_LOG_MAX>(g.lny, [&](auto c) -> cavity_status {
    constexpr int LN = decltype(c)::value;
    using F = F32Shape<LN>;
    static DeviceFlag done;
    const dim3 grid((g.nx + F::R - 1) / F::R, 2, ndir);
    if constexpr (F::R > 1 << CAV_LOG_MIN) {
      if (g.nx < F::R) {
        static DeviceFlag done1;
        CKS(smem_once(ctx, k_opA<LN, true>, done1));
        KScope ks_(ctx, KC_TBC_A32);
        k_opA<LN, true><<<grid, F::NT, SmemA<LN>::BYTES, st>>>(x, R1, p, ctx->lane_tab[1],
                                                              ctx->ehat_y32[0], ctx->ehat_y32[1]);
        return CAVITY_OK;
      }
    }
    CKS(smem_once(ctx, k_opA<LN, false>, done));
    KScope ks_(ctx, KC_TBC_A32);
    k_opA<LN, false><<<grid, F::NT, SmemA<LN>::BYTES, st>>>(x, R1, p, ctx->lane_tab[1],
                                                           ctx->ehat_y32[0], ctx->ehat_y32[1]);
    return CAVITY_OK;
  }));
  CKS(dispatch_log<CAV_LOG_MIN, CAV_LOG_MAX>(g.lnx, [&](auto c) -> cavity_status {
    constexpr int LN = decltype(c)::value;
    using F = F32Shape<LN>;
    static DeviceFlag done;
    CKS(smem_once(ctx, k_opB<LN>, done));
    KScope ks_(ctx, KC_TBC_B32);
    k_opB<LN><<<dim3(g.Py / F::CB, ndir), F::NT, SmemB<LN>::BYTES, st>>>(
        R1, R2, p, ctx->lane_tab[0], ctx->ehat_x32[0], ctx->ehat_x32[1], ctx->khat32s,
        (float)(2.0 * M_PI / g.Lx), (float)(2.0 * M_PI / g.Ly));
    return CAVITY_OK;
  }));
  CKS(dispatch_log<CAV_LOG_MIN, CAV_LOG_MAX>(g.lny, [&](auto c) -> cavity_status {
    constexpr int LN = decltype(c)::value;
    constexpr int R = SmemC<LN>::R;
    const dim3 grid((g.nx + 1 + R - 1) / R, 3, ndir);
    if (g.nx < 16) {
      static DeviceFlag done1;
      CKS(smem_once(ctx, k_opC<LN, true>, done1));
      KScope ks_(ctx, KC_TBC_C32);
      k_opC<LN, true><<<grid, SmemC<LN>::NT, SmemC<LN>::BYTES, st>>>(R2, R1, p, ctx->lane_tab[1]);
      return CAVITY_OK;
    }
    static DeviceFlag done;
    CKS(smem_once(ctx, k_opC<LN, false>, done));
    KScope ks_(ctx, KC_TBC_C32);
    k_opC<LN, false><<<grid, SmemC<LN>::NT, SmemC<LN>::BYTES, st>>>(R2, R1, p, ctx->lane_tab[1]);
    return CAVITY_OK;
  }));
  CKS(dispatch_log<CAV_LOG_MIN, CAV_LOG_MAX>(g.lnx, [&](auto c) -> cavity_status {
    constexpr int LN = decltype(c)::value;
    constexpr int R = SmemD<LN>::R;
    static DeviceFlag done;
    CKS(smem_once(ctx, k_opD<LN>, done));
    KScope ks_(ctx, KC_TBC_D32);
    k_opD<LN><<<dim3((g.ny + R - 1) / R, 3, ndir), SmemD<LN>::NT, SmemD<LN>::BYTES, st>>>(
        R1, R2, p, ctx->lane_tab[0]);
    return CAVITY_OK;
  }));
  {
    KScope ks_(ctx, KC_COMB32);
    k_combine<float><<<dim3((g.nx * g.ny + 255) / 256, ndir), 256, 0, st>>>(
        x, R2, ctx->top32, y, ystride, g.ny, p, last_m(ctx), last_n(ctx), pm);
  }
  CK(cudaGetLastError());
  return CAVITY_OK;
}
