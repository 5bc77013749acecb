// Interior field of the mixed path (complex64) on grids of 16 .. 1024
// intervals per side: back-substitution (EInter) and the syntheses (E123F) in
// two passes of register-resident line transforms (gfft.cuh).
//
// Per level j and direction, with c_l = P_l E_l (+ Q_l E_3):
//  pass Y, row m: the lines of E1 (sine in x2) and E2 (cosine) go through one
//    transform of length 2 ny as the odd and even part of a line,
//      z_n = c2 + c1,  z_{2ny-n} = c2 - c1,  z_0 = 2 c2:   Z = 2 C2 + 2 i S1;
//    E3 (sine) is the odd extension of its row:  Z3 = 2 i S3.
//  pass X, column q: E1 is the cosine and E2 the sine series along x1, and
//      y_m = Z(m, q),  y_{2nx-m} = -Z(m, -q),  y_0 = 2 Z(0, q)
//    is already the line whose transform is Y = 4 i (E1 + E2), E1 its even and
//    E2 its odd part in p: the two syntheses of pass Y are never separated.
//    E3 from the odd extension of Z3: Y3 = -4 E3.
// The intermediate is stored for its reader, [q][m] (whole lines of pass X),
// pass Y turning its rows through shared memory; pass X writes field rows 8
// columns at a time.  Chunks of 512 MB of intermediate: smaller ones that stay
// in L2 lose more to short grids than they save in traffic (512 x 512 x 256, 8
// directions: 16.2 ms at 64 MB, 13.1 at 256 MB, 12.5 at 512 MB).
// Bound: the shared-memory and L1 pipe (pass Y 75 %, X 65 % busy), then issue
// (46, 58 %) and DRAM (46, 56 %).  Measured on a GB300, whole field, before (a
// persistent kernel that kept the intermediate in L2 at 512 x 512, lines in
// shared memory elsewhere) and now:
//   512 x 512 x 256, 8 directions, 4 layers  20.6 -> 12.5 ms
//   256 x 256 x 128, 16 directions           5.44 -> 2.66 ms
//   256 x 128 x 91, 3 directions, 3 layers   0.47 -> 0.22 ms
//   64 x 64 x 32, 32 directions, 3 layers    0.25 -> 0.14 ms
#include <algorithm>

#include "common.cuh"
#include "gfft.cuh"

namespace {

struct FyP {
  int nx, ny, nz, M, N, n1, n2, nap;
  int j0, ndir;         // slabs s = (j - j0) ndir + d
  long long S;          // samples per level
};

// LN = log2 of the axis' intervals; lines of 2 << LN points
template <int LN, int NT> struct FShape {
  using S = GShape<LN + 1>;
  static constexpr int N2 = 2 << LN, LG = S::LG, RV = S::RV, H = RV / 2;
  static constexpr int R = NT / LG;                   // lines per block
  static constexpr int RAW = RV * (LG + 1);           // tile; holds the line, too
  // line pitch: the lines of a block, read column by column, on distinct banks
  static constexpr int LP = RAW / 16 * 16 + 16 + (R >= 16 ? 1 : 16 / R);
  static constexpr size_t BYTES = sizeof(float2) * (size_t)R * LP;
};
constexpr int FY_NT = 128, FX_NT = 256;

// ------------------------------------------------------------------ pass Y
// Coefficients of a row m at n = l + LG r, r < H, into the line's input.  The
// loads carry no branches (indices outside a component's set are clamped and
// their values dropped), so FY_BATCH values of r are in flight at once; with
// branches on the index sets the pass waited for memory 8 of 12 cycles
// (512 x 512, 48 slabs: 272 us, 170 us now).
#define FY_BATCH 4
template <int LNY, int KIND, bool LAY, int LG, int RV>
__device__ __forceinline__ void fy_load(float2 (&v)[RV], float2* line, const float2* __restrict__ E,
                                        const float2* __restrict__ P, const float2* __restrict__ Q,
                                        const FyP& p, int m, int l, bool in, bool top) {
  constexpr int H = RV / 2, ny = 1 << LNY, N = ny - 1, BT = H < FY_BATCH ? H : FY_BATCH;
  const int mr = min(m, p.nx - 1), m1 = max(mr, 1);
  const int i1 = mr * N - 1, i2 = p.n1 + (m1 - 1) * ny, i3 = p.n1 + p.n2 + (m1 - 1) * N - 1;
  const bool has = in && m >= 1;
  const float2 zero = make_float2(0.f, 0.f);
#pragma unroll
  for (int r0 = 0; r0 < H; r0 += BT) {
    float2 e1[BT], e2[BT], e3[BT], p1[BT], p2[BT], q1[BT], q2[BT];
#pragma unroll
    for (int b = 0; b < BT; ++b) {
      const int n = l + LG * (r0 + b), nn = max(n, 1);
      if constexpr (KIND == 0) {
        e1[b] = __ldg(E + i1 + nn);
        p1[b] = __ldg(P + i1 + nn);
        e2[b] = __ldg(E + i2 + n);
        p2[b] = __ldg(P + i2 + n);
        if constexpr (LAY) {
          e3[b] = __ldg(E + i3 + nn);
          q1[b] = __ldg(Q + i1 + nn);
          q2[b] = __ldg(Q + i2 + n);
        }
      } else {
        e3[b] = __ldg(E + i3 + nn);
        p1[b] = __ldg(P + i3 + nn);
      }
    }
#pragma unroll
    for (int b = 0; b < BT; ++b) {
      const int n = l + LG * (r0 + b);
      if constexpr (KIND == 0) {
        float2 c1 = cmul<float>(p1[b], e1[b]), c2 = cmul<float>(p2[b], e2[b]);
        if constexpr (LAY) {
          if (has && n >= 1) {
            c1 = cadd<float>(c1, cmul<float>(q1[b], e3[b]));
            c2 = cadd<float>(c2, cmul<float>(q2[b], e3[b]));
          }
        }
        if (top) {
          c1 = e1[b];
          c2 = e2[b];
        }
        if (!in || n < 1) c1 = zero;
        if (!has) c2 = zero;
        v[r0 + b] = n == 0 ? make_float2(2.f * c2.x, 2.f * c2.y) : cadd<float>(c2, c1);
        line[n] = csub<float>(c2, c1);
      } else {
        float2 c3 = top ? e3[b] : cmul<float>(p1[b], e3[b]);
        if (!has || n < 1) c3 = zero;
        v[r0 + b] = c3;
        line[n] = make_float2(-c3.x, -c3.y);
      }
    }
  }
}

// grid (ceil(nx / R), 2 kinds, slabs); kind 0: E1 with E2, 1: E3
template <int LNY, bool LAY>
__global__ void __launch_bounds__(FY_NT, 4)
    k_fy(const float2* __restrict__ ap, const float2* __restrict__ prof,
         const float2* __restrict__ profq, float2* __restrict__ T1, FyP p,
         const float2* __restrict__ lt) {
  using F = FShape<LNY, FY_NT>;
  constexpr int LG = F::LG, RV = F::RV, H = F::H, n2 = F::N2, ny = 1 << LNY;
  constexpr int R = F::R, LP = F::LP;
  extern __shared__ __align__(16) float2 smf[];
  const int kind = blockIdx.y, s = blockIdx.z, d = s % p.ndir, j = p.j0 + s / p.ndir;
  const int g = threadIdx.x / LG, l = threadIdx.x % LG;
  const int m0 = blockIdx.x * R, m = m0 + g;
  const bool top = j == p.nz, in = m < p.nx;
  float2* line = smf + g * LP;
  const float2* E = ap + (size_t)d * p.nap;
  const int jl = top ? 0 : j - 1;   // the aperture level has no profile
  const float2* P = prof + (size_t)jl * p.nap;
  const float2* Q = LAY ? profq + (size_t)jl * (p.n1 + p.n2) : nullptr;
  float2 v[RV];
  if (kind == 0) fy_load<LNY, 0, LAY, LG, RV>(v, line, E, P, Q, p, m, l, in, top);
  else fy_load<LNY, 1, LAY, LG, RV>(v, line, E, P, Q, p, m, l, in, top);
  group_sync<LG>(1 + g);
#pragma unroll
  for (int r = H; r < RV; ++r) {
    const int n = n2 - (l + LG * r);     // 1 .. ny
    v[r] = n < ny ? line[n] : make_float2(0.f, 0.f);
  }
  group_sync<LG>(1 + g);
  gfft<true, LG, RV>(v, line, l, lt, 1 + g);
  // rows of the block, consecutive m together; E3 needs 0 <= q < ny only
  float2* dst = T1 + (size_t)s * 3 * p.nx * ny + (kind ? (size_t)n2 * p.nx : 0) + m0;
#pragma unroll
  for (int r = 0; r < RV; ++r)
    if (kind == 0 || r < H) line[l + LG * r] = v[r];
  __syncthreads();
  const int nq = kind == 0 ? n2 : ny;
#pragma unroll 4
  for (int i = threadIdx.x; i < nq * R; i += FY_NT) {
    const int row = i % R, q = i / R;
    if (m0 + row < p.nx) dst[(size_t)q * p.nx + row] = smf[row * LP + q];
  }
}

// ------------------------------------------------------------------ pass X
// grid (ceil((ny + 1) / R), 2 kinds, slabs)
template <int LNX>
__global__ void __launch_bounds__(FX_NT, 2)
    k_fx(const float2* __restrict__ T1, float2* __restrict__ out, FyP p,
         const float2* __restrict__ lt) {
  using F = FShape<LNX, FX_NT>;
  constexpr int LG = F::LG, RV = F::RV, H = F::H, n2 = F::N2, nx = 1 << LNX;
  constexpr int R = F::R, LP = F::LP;
  extern __shared__ __align__(16) float2 smf[];
  const int kind = blockIdx.y, s = blockIdx.z, d = s % p.ndir, j = p.j0 + s / p.ndir, ny = p.ny;
  const int g = threadIdx.x / LG, l = threadIdx.x % LG;
  const int q0 = blockIdx.x * R, q = q0 + g;
  if (kind == 1 && q0 >= ny) return;     // uniform over the block
  float2* line = smf + g * LP;
  const float2* t1 = T1 + (size_t)s * 3 * nx * ny + (kind ? (size_t)2 * ny * nx : 0);
  const bool in = kind ? q < ny : q <= ny;
  const float2* a = t1 + (size_t)(in ? q : 0) * nx;
  const float2* b = kind ? a : t1 + (size_t)(in && q > 0 ? 2 * ny - q : 0) * nx;
  const float2 zero = make_float2(0.f, 0.f);
  float2 v[RV];
#pragma unroll
  for (int r = 0; r < H; ++r) {
    const int m = l + LG * r;
    float2 c = a[m];
    if (m == 0) c = kind ? zero : make_float2(2.f * c.x, 2.f * c.y);
    v[r] = c;
    const int mm = LG * (H - r) - l;       // mirrored slot r + H: 1 .. nx
    c = mm < nx ? b[mm] : zero;
    v[r + H] = make_float2(-c.x, -c.y);
  }
  gfft<true, LG, RV>(v, line, l, lt, 1 + g);
#pragma unroll
  for (int r = 0; r < RV; ++r)
    if (kind == 0 || r < H) line[l + LG * r] = v[r];
  __syncthreads();
  float2* o = out + ((size_t)d * p.nz + (j - 1)) * p.S;
  const long long offE2 = (long long)(nx + 1) * (ny - 1);
  const long long offE3 = offE2 + (long long)(nx - 1) * (ny + 1);
  if (kind == 0) {
    for (int i = threadIdx.x; i < (nx + 1) * R; i += FX_NT) {
      const int c = i % R, pp = i / R, qc = q0 + c;
      if (qc > ny) continue;
      const float2 w = smf[c * LP + pp], u = smf[c * LP + ((n2 - pp) & (n2 - 1))];
      // 1 / (8 i): (x, y) -> (y, -x) / 8
      if (qc >= 1 && qc < ny)
        __stcs(o + (size_t)pp * (ny - 1) + (qc - 1),
               make_float2(0.125f * (w.y + u.y), -0.125f * (w.x + u.x)));
      if (pp >= 1 && pp < nx)
        __stcs(o + offE2 + (size_t)(pp - 1) * (ny + 1) + qc,
               make_float2(0.125f * (w.y - u.y), -0.125f * (w.x - u.x)));
    }
  } else {
    for (int i = threadIdx.x; i < (nx - 1) * R; i += FX_NT) {
      const int c = i % R, pp = 1 + i / R, qc = q0 + c;
      if (qc < 1 || qc >= ny) continue;
      const float2 w = smf[c * LP + pp];
      __stcs(o + offE3 + (size_t)(pp - 1) * (ny - 1) + (qc - 1), make_float2(-0.25f * w.x, -0.25f * w.y));
    }
  }
}

template <typename K> cavity_status smem_set(cavity_ctx* ctx, K kern, DeviceFlag& done) {
  if (!done) {
    CK(allow_max_smem(kern));
    done.set();
  }
  return CAVITY_OK;
}

}  // namespace

bool field_f32_supported(const Geo& g) {
  return g.lnx >= FIELD_F32_LOG_MIN && g.lny >= FIELD_F32_LOG_MIN;
}
size_t field_f32_slab_bytes(const Geo& g) { return sizeof(float2) * 3 * (size_t)g.nx * g.ny; }

// levels j0 .. j0 + nlev - 1 of all directions; T1: slab bytes x ndir x nlev
cavity_status launch_field_f32(cavity_ctx* ctx, int ndir, const float2* ap, float2* out, float2* T1,
                               int j0, int nlev) {
  const Geo& g = ctx->g;
  FyP p;
  p.nx = g.nx; p.ny = g.ny; p.nz = g.nz; p.M = g.M; p.N = g.N; p.n1 = g.n1; p.n2 = g.n2;
  p.nap = g.nap; p.j0 = j0; p.ndir = ndir; p.S = g.field_per_level;
  const float2* profq = ctx->layers.size() > 1 ? ctx->profq32 : nullptr;
  CKS(dispatch_log<FIELD_F32_LOG_MIN, CAV_LOG_MAX>(g.lny, [&](auto c) -> cavity_status {
    constexpr int LN = decltype(c)::value;
    using F = FShape<LN, FY_NT>;
    static DeviceFlag done[2];
    const dim3 grid((g.nx + F::R - 1) / F::R, 2, ndir * nlev);
    CKS(smem_set(ctx, k_fy<LN, false>, done[0]));
    CKS(smem_set(ctx, k_fy<LN, true>, done[1]));
    KScope ks_(ctx, KC_FIELD_Y);
    if (profq)
      k_fy<LN, true><<<grid, FY_NT, F::BYTES, ctx->stream>>>(ap, ctx->prof32, profq, T1, p,
                                                            ctx->lane_tab_f[1]);
    else
      k_fy<LN, false><<<grid, FY_NT, F::BYTES, ctx->stream>>>(ap, ctx->prof32, nullptr, T1, p,
                                                             ctx->lane_tab_f[1]);
    return CAVITY_OK;
  }));
  CKS(dispatch_log<FIELD_F32_LOG_MIN, CAV_LOG_MAX>(g.lnx, [&](auto c) -> cavity_status {
    constexpr int LN = decltype(c)::value;
    using F = FShape<LN, FX_NT>;
    static DeviceFlag done;
    CKS(smem_set(ctx, k_fx<LN>, done));
    KScope ks_(ctx, KC_FIELD_X);
    k_fx<LN><<<dim3((g.ny + F::R) / F::R, 2, ndir * nlev), FX_NT, F::BYTES, ctx->stream>>>(
        T1, out, p, ctx->lane_tab_f[0]);
    return CAVITY_OK;
  }));
  CK(cudaGetLastError());
  return CAVITY_OK;
}
