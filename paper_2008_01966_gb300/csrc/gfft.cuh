// Register-resident FP32 transforms by groups of lanes, for the passes of the
// FP32 operator (tbc_f32.cu) and of the complex64 field (field_f32.cu).
//
// A group of LG lanes (4 .. 128) holds a line of n = LG RV points, RV values
// per lane, lane l holding x[l + LG r].  The transform is one register DFT of
// RV points, the twiddle w_n^{l k1}, one transpose through shared memory, and
// a DFT of LG points, and it returns its result in the SAME distribution,
// v[s] = X[l + LG s]: a product with a table in the frequency domain and the
// next transform need no further pass through shared memory.  One transform
// moves every value through shared memory twice (one write, one read; C reads
// where C = LG / RV > 1 lanes share a DFT of the second stage, see below),
// where a transform with lines in shared memory moves it four to five times;
// that pipe is what bounded the operator passes.
//
// Second stage: the RV rows k1 of the tile (pitch LG + 1) are transformed over
// l.  LG <= RV: lane l takes the rows l + LG q, q < RV / LG.  LG > RV: the C
// lanes l = k1 + RV h, h < C, share row k1; lane h folds the row by radix C,
//   u[l'] = w_LG^{h l'} sum_q w_C^{h q} a[l' + RV q],   l' < RV,
// and its RV-point DFT gives X[k1 + RV (C s + h)] = X[l + LG s].
//
// Twiddles are read from per-length tables laid out by lane (LaneTab): the
// lanes of a warp read consecutive words.  With the strided reads of one
// shared table the twiddle loads took more of the L1 pipe than the data.
#pragma once
#include "fft.cuh"

// lanes and values per lane of a line of 2^LOGN points
template <int LOGN> struct GShape {
  static_assert(LOGN >= 4 && LOGN <= 12, "lines of 16 to 4096 points");
  static constexpr int RV = LOGN >= 9 ? 32 : 1 << ((LOGN + 1) / 2);
  static constexpr int LG = (1 << LOGN) / RV;
};
// tile of one group (elements): the stride between the groups of a warp keeps
// 16 consecutive lanes on distinct banks
template <int LG, int RV> struct GTile {
  static constexpr int PITCH = LG + 1;
  static constexpr int RAW = RV * PITCH;
  static constexpr int SIZE = LG == 8 ? RAW + ((24 - RAW % 16) % 16) : RAW;
};

// lane table of one grid axis with n = 2^LOGN: [w_n^{l k1}] (k1-major, LG
// wide), fold factors [w_LG^{h l'}] (h-major, RV wide; LG entries), the same
// two for n/2 points (RV/2 values per lane), and exp(+2 pi i p / n), p <= n/4.
__host__ __device__ constexpr int lane_tab_half(int n, int LG) { return n + LG; }
__host__ __device__ constexpr int lane_tab_post(int n, int LG) { return n + LG + n / 2 + LG; }
__host__ __device__ constexpr int lane_tab_size(int n, int LG) {
  return lane_tab_post(n, LG) + n / 4 + 1;
}

// 4-point DFT of (a0, 0, 0, a3)
template <bool INV>
__device__ __forceinline__ void dft4sz(float2* v, int st) {
  const float2 a0 = v[0], a3 = v[3 * st];
  const float2 e = mulmi<float, INV>(a3);
  v[0] = cadd<float>(a0, a3);
  v[2 * st] = csub<float>(a0, a3);
  v[st] = csub<float>(a0, e);
  v[3 * st] = cadd<float>(a0, e);
}
// DFT of R points whose middle half (R/4 <= r < 3R/4) is zero: the first
// radix-4 step has two inputs instead of four
template <bool INV>
__device__ __forceinline__ void dft16z(float2* v) {
#pragma unroll
  for (int c = 0; c < 4; ++c) dft4sz<INV>(v + c, 4);
  const float c1 = (float)FFT_C16, s1 = (float)FFT_S16, c2 = (float)FFT_C8;
  v[5] = mulw<float, INV>(v[5], c1, s1);
  v[9] = mulw<float, INV>(v[9], c2, c2);
  v[13] = mulw<float, INV>(v[13], s1, c1);
  v[6] = mulw<float, INV>(v[6], c2, c2);
  v[10] = mulmi<float, INV>(v[10]);
  v[14] = mulw<float, INV>(v[14], -c2, c2);
  v[7] = mulw<float, INV>(v[7], s1, c1);
  v[11] = mulw<float, INV>(v[11], -c2, c2);
  v[15] = mulw<float, INV>(v[15], -c1, -s1);
#pragma unroll
  for (int r = 0; r < 4; ++r) dft4s<float, INV>(v + 4 * r, 1);
}
template <bool INV, int R>
__device__ __forceinline__ void dft_natz(float2* v) {
  if constexpr (R == 4) {
    dft4sz<INV>(v, 1);
  } else if constexpr (R == 8) {
    float2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    dft4sz<INV>(e, 1);
    dft4sz<INV>(o, 1);
    const float c = (float)FFT_C8;
    o[1] = mulw<float, INV>(o[1], c, c);
    o[2] = mulmi<float, INV>(o[2]);
    o[3] = mulw<float, INV>(o[3], -c, c);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = cadd<float>(e[k], o[k]);
      v[k + 4] = csub<float>(e[k], o[k]);
    }
  } else if constexpr (R == 16) {
    float2 u[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) u[i] = v[i];
    dft16z<INV>(u);
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = u[dft16_slot(k)];
  } else {
    static_assert(R == 32, "4, 8, 16 or 32 values per lane");
    float2 e[16], o[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      e[i] = v[2 * i];
      o[i] = v[2 * i + 1];
    }
    dft16z<INV>(e);
    dft16z<INV>(o);
    const float cs[16] = {1.0f, (float)0.98078528040323044913, (float)0.92387953251128675613,
                          (float)0.83146961230254523708, (float)0.70710678118654752440,
                          (float)0.55557023301960222474, (float)0.38268343236508977173,
                          (float)0.19509032201612826785, 0.0f, (float)-0.19509032201612826785,
                          (float)-0.38268343236508977173, (float)-0.55557023301960222474,
                          (float)-0.70710678118654752440, (float)-0.83146961230254523708,
                          (float)-0.92387953251128675613, (float)-0.98078528040323044913};
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float c = cs[k], sn = cs[k < 8 ? 8 - k : k - 8];
      const float2 t = mulw<float, INV>(o[dft16_slot(k)], c, sn);
      const float2 ev = e[dft16_slot(k)];
      v[k] = cadd<float>(ev, t);
      v[k + 16] = csub<float>(ev, t);
    }
  }
}

// barrier of the LG lanes of one group (LG > 32: the named barrier `bar`)
template <int LG> __device__ __forceinline__ void group_sync(int bar) {
  if constexpr (LG <= 32) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(LG) : "memory");
}

// multiply by w or conj(w) (tables hold the forward factors)
template <bool INV> __device__ __forceinline__ float2 cmul_tw(float2 v, float2 w) {
  return INV ? make_float2(v.x * w.x + v.y * w.y, v.y * w.x - v.x * w.y) : cmul<float>(v, w);
}

// The group transform.  lt: [w_n^{l k1}] then the fold factors (LaneTab parts
// of this length).  ZMID: the inputs r in [RV/4, 3RV/4) are zero.  All lanes
// of the group call; the tile is free again on return.
template <bool INV, int LG, int RV, bool ZMID = false>
__device__ __forceinline__ void gfft(float2 (&v)[RV], float2* tile, int l,
                                     const float2* __restrict__ lt, int bar) {
  constexpr int PITCH = LG + 1;
  if constexpr (ZMID) dft_natz<INV, RV>(v);
  else dft_nat<float, INV, RV>(v);
  tile[l] = v[0];
#pragma unroll
  for (int k1 = 1; k1 < RV; ++k1) tile[k1 * PITCH + l] = cmul_tw<INV>(v[k1], __ldg(lt + k1 * LG + l));
  group_sync<LG>(bar);
  if constexpr (LG <= RV) {
    constexpr int Q = RV / LG;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      float2 u[LG];
#pragma unroll
      for (int i = 0; i < LG; ++i) u[i] = tile[(l + LG * q) * PITCH + i];
      dft_nat<float, INV, LG>(u);
#pragma unroll
      for (int k2 = 0; k2 < LG; ++k2) v[q + Q * k2] = u[k2];
    }
  } else {
    constexpr int C = LG / RV;
    const int k1 = l & (RV - 1), h = l / RV;
    const float2* row = tile + k1 * PITCH;
    const float2* fold = lt + LG * RV + h * RV;
    const float e = (h & 1) ? -1.f : 1.f;   // w_C^{h C/2}
    if constexpr (C == 2) {
#pragma unroll
      for (int i = 0; i < RV; ++i) {
        const float2 a = row[i], b = row[i + RV];
        v[i] = cmul_tw<INV>(make_float2(fmaf(e, b.x, a.x), fmaf(e, b.y, a.y)), __ldg(fold + i));
      }
    } else if constexpr (C == 4) {
      // w_4^h: (1, -i, -1, i) forward
      const float cr = (h & 1) ? 0.f : (h == 0 ? 1.f : -1.f);
      float ci = (h & 1) ? (h == 1 ? -1.f : 1.f) : 0.f;
      if (INV) ci = -ci;
#pragma unroll
      for (int i = 0; i < RV; ++i) {
        const float2 a = row[i], b = row[i + RV], c = row[i + 2 * RV], d = row[i + 3 * RV];
        const float2 y0 = make_float2(fmaf(e, c.x, a.x), fmaf(e, c.y, a.y));
        const float2 y1 = make_float2(fmaf(e, d.x, b.x), fmaf(e, d.y, b.y));
        const float2 u = make_float2(fmaf(cr, y1.x, fmaf(-ci, y1.y, y0.x)),
                                     fmaf(cr, y1.y, fmaf(ci, y1.x, y0.y)));
        v[i] = cmul_tw<INV>(u, __ldg(fold + i));
      }
    } else {
      static_assert(C == 8, "two, four or eight lanes per second-stage DFT");
      // w_8^{h q}, q = 1, 2, 3
      const float r2 = (float)FFT_C8;
      const float cx[8] = {1.f, r2, 0.f, -r2, -1.f, -r2, 0.f, r2};
      float2 w[3];
#pragma unroll
      for (int q = 1; q < 4; ++q) {
        const int k = (h * q) & 7;
        float c = 1.f, s = 0.f;   // cos, sin of 2 pi k / 8
#pragma unroll
        for (int t = 0; t < 8; ++t)
          if (k == t) {
            c = cx[t];
            s = cx[(t + 6) & 7];
          }
        w[q - 1] = make_float2(c, INV ? s : -s);
      }
#pragma unroll
      for (int i = 0; i < RV; ++i) {
        float2 u = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 a = row[i + q * RV], b = row[i + (q + 4) * RV];
          const float2 y = make_float2(fmaf(e, b.x, a.x), fmaf(e, b.y, a.y));
          if (q == 0) u = y;
          else u = cadd<float>(u, cmul<float>(y, w[q - 1]));
        }
        v[i] = cmul_tw<INV>(u, __ldg(fold + i));
      }
    }
    dft_nat<float, INV, RV>(v);
  }
  group_sync<LG>(bar);
}
