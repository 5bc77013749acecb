// Block GMRES in FP32 for the inner solves of the mixed-precision refinement.
//
// All incident directions of a solve share the operator, so their Krylov
// spaces are built together (block Arnoldi): the directions are split into
// groups of at most BG_MAX, and step k of a group extends its basis by the
// block A M^{-1} V_k of all its directions at once.  A direction's correction
// is then sought in the whole block space, which contains its own
// single-direction Krylov space of the same step count; the block solve reaches
// the inner tolerance in fewer operator applications (measured with the oracle
// on the 16-direction 64^2 and 128^2 workloads: 10-11 block steps against
// 13-14 per-direction steps to 1e-5).
//
// Orthogonalisation of the new block W against the basis V: one classical
// Gram-Schmidt pass as two GEMM-shaped tensor-core kernels, TF32 operands
// split into three products for FP32 accuracy.  (Blocks of few columns
// take kernels on the FP32 lanes, further down.)  W -= V H (k_bnn_tc5) runs on
// the fifth-generation tensor cores (tcgen05.mma kind::tf32, accumulators in
// tensor memory; tc05.cuh).  V^H W is a split reduction over the rows
// (k_bproj_tc, then k_bproj_final in a fixed order) on warp-level mma.sync: a
// tcgen05 version measured 2x slower, its threads having to split and place
// every element in the core-matrix layout of the reduction dimension, where
// the mma.sync version splits fragments in registers from tiles staged by
// cp.async.  The Gram matrix of the projected block is then formed
// (k_bproj_tc with W against itself) and the block is
// orthonormalised by Cholesky QR, or by SVQB (Stathopoulos and Wu, 2002:
// W = V' S with V' = W U Lambda^{-1/2} from G = W^H W = U Lambda U^H,
// eigenvalues below a floor raised to it) when it is nearly dependent
// (repeated incident directions, converged columns), so W = V' S holds
// exactly and nothing divides by ~0; a vanished block is an exact breakdown.
//
// The least-squares problems min || E_1 S_0 - Hbar Y || (block upper Hessenberg,
// one right-hand side per direction of the group) are solved on the host in
// FP64 by Householder reflections, one new column at a time; the norm of the
// tail of each transformed right-hand side is that direction's residual.
//
// Reductions are fixed-order trees, so the result is deterministic for a given
// batch; unlike per-direction GMRES it depends (within the tolerance) on which
// directions share a group.
#include <algorithm>
#include <cmath>
#include <complex>
#include <vector>

#include "bgmres_host.h"
#include "common.cuh"
#include "tc05.cuh"

#define BG_GROUPS 32      // groups per call (BG_GROUPS * BG_MAX directions)
#define BG_PART_CTAS 608  // bound on groups x row chunks of one projection

#define BG_CLASSES 4      // parity classes (ParityMap), each a system of its own

// One system of a call: a parity class of a group of directions (all classes
// in one when the order of Appendix A is kept).
struct BGrp {
  const float2* V;  // Kv basis columns, stride nap
  const float2* W;  // r block columns, stride nap
  float2* O;        // output columns, stride nap (k_bnn_tc5)
  int n;            // rows
  int Kv;           // columns taken from V (k_bnn_tc5 multiplies these)
  int K;            // projected columns (k_bproj_tc): V_0..V_{Kv-1}, then W_0..W_{K-Kv-1}
  int r;
  int coff;         // offset of this group's coefficient matrix (BG_MAX wide)
};
struct BGSet {
  BGrp g[BG_GROUPS * BG_CLASSES];
};

// a second Gram-Schmidt pass where the orthonormalising transform magnified a
// block's rounding by more than this (measured: at 20 some classes still
// stalled, at 10 few, at 5 none; every class of every step costs 2-5 % more)
#define BG_REORTH 5.0
#define BG_REORTH_FULL 3e3
#define BP_ROWS 128  // rows per staged tile (slabs are whole tiles)

__device__ __forceinline__ void cp_async8(float2* dst, const float2* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = valid ? 8 : 0;  // 0: the 8 bytes are zero-filled
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(n));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

// h[z][i][j] = sum over the nct slabs of part[z][x][i][j] in a fixed order.
// grid (K, groups), 256 threads: thread t adds the slabs x = t >> 4 (mod 16)
// of column j = t & 15 (16 consecutive threads read one 256-byte row of
// partials), and the 16 slab classes are added in class order.
__global__ void __launch_bounds__(256) k_bproj_final(BGSet set, const double2* __restrict__ part,
                                                     double2* __restrict__ h, int nct, int kcap) {
  __shared__ double2 q16[16][16];
  const BGrp& gd = set.g[blockIdx.y];
  const int i = blockIdx.x;
  if (i >= gd.K) return;  // uniform over the block
  const int t = threadIdx.x, j = t & 15, xg = t >> 4;
  double sx = 0, sy = 0;
  if (j < gd.r) {
#pragma unroll 4
    for (int x = xg; x < nct; x += 16) {
      const double2 v = part[((size_t)(blockIdx.y * nct + x) * kcap + i) * BG_MAX + j];
      sx += v.x;
      sy += v.y;
    }
  }
  q16[xg][j] = make_double2(sx, sy);
  __syncthreads();
  if (t < 16 && t < gd.r) {
    double ax = 0, ay = 0;
#pragma unroll
    for (int q = 0; q < 16; ++q) { ax += q16[q][t].x; ay += q16[q][t].y; }
    h[((size_t)blockIdx.y * kcap + i) * BG_MAX + t] = make_double2(ax, ay);
  }
}

// Block update: O_j[e] = beta W_j[e] + sgn sum_{i<Kv} V_i[e] C[i][j] for j < r
// (C: the group's coefficient matrix at cmat + coff, FP64, BG_MAX wide).  The
// complex product is a real GEMM,
//   [Re O_j, Im O_j] = sum_i [Re V_i, Im V_i] [[Re C_ij, Im C_ij], [-Im C_ij, Re C_ij]],
// of n_ap rows, 2 Kv inner terms and 32 outputs.
// It runs on the fifth-generation tensor cores (tcgen05.mma
// kind::tf32, accumulator in tensor memory; layouts and the TF32 split in
// tc05.cuh): grid (ceil(nap / 128), 1, groups), 128 threads (one warpgroup),
// the block's 128 rows x 32 real outputs in 32 columns of tensor memory.
// Chunks of T5_CH = 8 complex basis columns (16 real inner terms, two MMA
// k-steps, three products each) pass through two shared-memory buffers: the
// threads stage chunk c + 1 while the tensor cores multiply chunk c.  The
// products hi hi and the two corrections go to separate accumulators (32
// columns each), drained into FP32 registers every TC_DRAIN chunks (see
// tc05.cuh).  Thread
// t stages row row0 + t of V (eight 8-byte loads, one per column, a warp's
// 32 rows contiguous) and one complex coefficient (u, j) = (t / 16, t % 16)
// as its 2 x 2 real block.  A wait that runs out sets *err and skips the
// output.
#define T5_CH 8
struct T5Buf {
  float a_hi[2][128 * 8], a_lo[2][128 * 8];  // [k-step][K-major tile]
  float b_hi[2][32 * 8], b_lo[2][32 * 8];
};
__device__ int g_tc_err;  // set when a tensor-core wait ran out

__global__ void __launch_bounds__(128) k_bnn_tc5(BGSet set, const double2* __restrict__ cmat,
                                                 int nap, float beta, float sgn) {
  extern __shared__ __align__(128) unsigned char t5raw[];
  T5Buf* bufs = (T5Buf*)t5raw;
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ uint32_t tslot;
  const BGrp& gd = set.g[blockIdx.z];
  const double2* Cm = cmat + gd.coff;
  const int Kv = gd.Kv, r = gd.r;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int row0 = blockIdx.x * 128, e = row0 + tid, nrow = gd.n;
  if (row0 >= nrow) return;  // uniform over the block
  const int nch = (Kv + T5_CH - 1) / T5_CH;
  if (nch == 0) {  // uniform over the block: O = beta O
    if (e < nrow)
      for (int j = 0; j < r; ++j) {
        const float2 ov = beta != 0.f ? gd.W[(size_t)j * nap + e] : make_float2(0.f, 0.f);
        gd.O[(size_t)j * nap + e] = make_float2(beta * ov.x, beta * ov.y);
      }
    return;
  }
  if (tid == 0) {
    tc_mbar_init(&mbar[0]);
    tc_mbar_init(&mbar[1]);
  }
  if (warp == 0) tc_alloc(&tslot, 64);
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  const uint32_t tmem = tslot;
  constexpr uint32_t idesc = tc_idesc_tf32(128, 32);
  bool ok = true;
  int last = -1;   // the last chunk whose MMAs were committed
  float racc[32];
#pragma unroll
  for (int n = 0; n < 32; ++n) racc[n] = 0.f;
  float2 v[T5_CH];
  double2 cnext;
  auto load_chunk = [&](int cn) {
#pragma unroll
    for (int u = 0; u < T5_CH; ++u) {
      const int i = cn * T5_CH + u;
      v[u] = (i < Kv && e < nrow) ? gd.V[(size_t)i * nap + e] : make_float2(0.f, 0.f);
    }
    const int iu = cn * T5_CH + (tid >> 4), j = tid & 15;
    cnext = (iu < Kv && j < r) ? Cm[(size_t)iu * BG_MAX + j] : make_double2(0.0, 0.0);
  };
  load_chunk(0);
  for (int c = 0; c < nch && ok; ++c) {
    const int b = c & 1;
    T5Buf& B = bufs[b];
    // the MMAs of chunk c - 2 read this buffer
    if (c >= 2) ok = tc_mbar_wait(&mbar[b], ((c - 2) >> 1) & 1);
    ok = __syncthreads_and(ok);
    if (!ok) break;
    // A: row tid, complex columns i = c T5_CH + u -> real inner terms 2u, 2u + 1
    // (values loaded one iteration ahead)
#pragma unroll
    for (int u = 0; u < T5_CH; ++u) {
      uint32_t hr, lr, hi, li;
      tc_split(v[u].x, hr, lr);
      tc_split(v[u].y, hi, li);
      const int ks = u >> 2, k8 = (2 * u) & 7, off = tc_koff(tid, k8);
      *(uint2*)((char*)B.a_hi[ks] + off) = make_uint2(hr, hi);
      *(uint2*)((char*)B.a_lo[ks] + off) = make_uint2(lr, li);
    }
    // B (N x K, K-major): real rows n = 2j + c' against inner terms k = 2u + c
    {
      const int u = tid >> 4, j = tid & 15;
      const double2 cc = cnext;
      if (c + 1 < nch) load_chunk(c + 1);   // in flight during the barrier and the MMAs
      const float cr = (float)(sgn * cc.x), ci = (float)(sgn * cc.y);
      const int ks = u >> 2, k8 = (2 * u) & 7;
      uint32_t h0, l0, h1, l1, h2, l2;
      tc_split(cr, h0, l0);
      tc_split(ci, h1, l1);
      tc_split(-ci, h2, l2);
      // (n = 2j: k = 2u -> cr, k = 2u + 1 -> -ci), (n = 2j + 1: ci, cr)
      *(uint2*)((char*)B.b_hi[ks] + tc_koff(2 * j, k8)) = make_uint2(h0, h2);
      *(uint2*)((char*)B.b_lo[ks] + tc_koff(2 * j, k8)) = make_uint2(l0, l2);
      *(uint2*)((char*)B.b_hi[ks] + tc_koff(2 * j + 1, k8)) = make_uint2(h1, h0);
      *(uint2*)((char*)B.b_lo[ks] + tc_koff(2 * j + 1, k8)) = make_uint2(l1, l0);
    }
    tc_fence_smem();
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    if (tid == 0) {
#pragma unroll
      for (int ks = 0; ks < 2; ++ks) {
        const uint64_t ah = tc_desc(B.a_hi[ks]), al = tc_desc(B.a_lo[ks]);
        const uint64_t bh = tc_desc(B.b_hi[ks]), bl = tc_desc(B.b_lo[ks]);
        const uint32_t acc = (c % TC_DRAIN != 0 || ks > 0) ? 1u : 0u;
        tc_mma(tmem, ah, bh, idesc, acc);         // hi hi
        tc_mma(tmem + 32, al, bh, idesc, acc);    // the corrections apart
        tc_mma(tmem + 32, ah, bl, idesc, 1u);
      }
      tc_commit(&mbar[b]);
    }
    last = c;
    if (c % TC_DRAIN == TC_DRAIN - 1 || c == nch - 1) {
      ok = __syncthreads_and(tc_mbar_wait(&mbar[b], (c >> 1) & 1));
      tc_after_sync();
      if (ok) tc_drain(tmem + ((uint32_t)(32 * warp) << 16), racc);
      tc_before_sync();
      __syncthreads();
    }
  }
  // every MMA done: the last chunk was drained
  if (ok) {
    const float* d = racc;
    if (e < nrow) {
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        if (j >= r) break;
        const float2 ov = beta != 0.f ? gd.W[(size_t)j * nap + e] : make_float2(0.f, 0.f);
        gd.O[(size_t)j * nap + e] =
            make_float2(beta * ov.x + d[2 * j], beta * ov.y + d[2 * j + 1]);
      }
    }
  } else if (tid == 0) {
    atomicExch(&g_tc_err, 1);
    tc_settle(mbar, last);   // MMAs in flight end before the tensor memory is freed
  }
  tc_before_sync();
  __syncthreads();
  if (warp == 0) tc_dealloc(tmem, 64);
}

__device__ __forceinline__ unsigned tf32_of(float x) {
  unsigned r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void tf32_split(float x, unsigned& hi, unsigned& lo) {
  hi = tf32_of(x);
  lo = tf32_of(x - __uint_as_float(hi));
}
// D += A B for one 16 x 8 x 8 tile; fragments as in the PTX ISA for .tf32:
// lane = 4 g + t; a0 (g, t), a1 (g + 8, t), a2 (g, t + 4), a3 (g + 8, t + 4);
// b0 (t, g), b1 (t + 4, g); d0 (g, 2t), d1 (g, 2t + 1), d2 (g + 8, 2t), d3 (g + 8, 2t + 1)
__device__ __forceinline__ void mma_tf32(float (&d)[4], const unsigned (&a)[4], unsigned b0,
                                         unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Partial projections: part[z][x][i][j] = sum over the rows e of slab x of
// conj(X_i[e]) W_j[e] for group z, i < K, j < r, where X_i is basis column i
// for i < Kv and block column i - Kv after that, on the tensor pipe.
// With real columns m = 2 i + c of V (component c of column i) and n = 2 j + c'
// of W, the real product P = Vr^T Wr over the rows of a slab gives
//   Re H_ij = P(2i, 2j) + P(2i+1, 2j+1),   Im H_ij = P(2i, 2j+1) - P(2i+1, 2j)
// (H = V^H W), with the three-product TF32 split.  grid (nslab,
// ceil(K / 16), groups), 128 threads: the block owns 16 complex V columns (32
// real rows of P, two m16 tiles) against all 16 W columns (32 real, four n8
// tiles) over its slab, walked in 64-row tiles staged by cp.async into two
// buffers (row pitch 40 words: the fragment loads of a warp hit distinct
// banks); warp w takes rows 16 w .. 16 w + 15 of each tile, and the four
// warps' sums are added in warp order at the end.
// NT: n8 tiles of W computed, 4 columns each: 2 where no group has more than 8
// columns (512 x 512, 8 directions: 4.16 -> 3.84 ms a solve), else 4.
#define TP_ROWS 64
#define TP_LD 40
#define TP_SMEM (sizeof(float) * 2 * 2 * TP_ROWS * TP_LD)
template <int NT>
__global__ void __launch_bounds__(128, 4) k_bproj_tc(BGSet set, double2* __restrict__ part, int nap,
                                                  int rs, int nct, int kcap) {
  extern __shared__ __align__(16) float tsm[];  // [buf][V | W][row][TP_LD]
  const BGrp& gd = set.g[blockIdx.z];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;
  const int ib = blockIdx.y * 16, K = gd.K, Kv = gd.Kv, r = gd.r;
  const int e0 = blockIdx.x * rs, e1 = min(gd.n, e0 + rs);
  // staging: element q = tid + 128 u (u < 8) of a 64 x 16 tile has row bits
  // 0-1 from q bits 0-1 and bits 2-5 from q bits 6-9, column q bits 2-5; a
  // half-warp writes 4 rows x 4 columns (distinct banks at the 40-word pitch)
  // and a warp reads 8 whole 32-byte sectors
  auto stage = [&](int buf, int eb) {
    float* vs = tsm + (size_t)buf * 2 * TP_ROWS * TP_LD;
    float* ws = vs + TP_ROWS * TP_LD;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int q = tid + 128 * u, c = (q >> 2) & 15, el = (q & 3) | ((q >> 6) << 2);
      const int e = eb + el, i = ib + c;
      const bool in = e < e1;
      const float2* src = i < Kv ? gd.V + (size_t)i * nap : gd.W + (size_t)(i - Kv) * nap;
      cp_async8((float2*)(vs + el * TP_LD + 2 * c), (in && i < K) ? src + e : gd.W, in && i < K);
    }
#pragma unroll
    for (int u = 0; u < 2 * NT; ++u) {   // 4 NT columns of W, row bits 2-5 from the top bits of q
      const int q = tid + 128 * u, c = (q >> 2) & (4 * NT - 1), el = (q & 3) | ((q / (16 * NT)) << 2);
      const int e = eb + el;
      const bool in = e < e1 && c < r;
      cp_async8((float2*)(ws + el * TP_LD + 2 * c), in ? gd.W + (size_t)c * nap + e : gd.W, in);
    }
    cp_async_commit();
  };
  float acc[2][NT][4];
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[mt][nt][q] = 0.f;
  const int ntile = (e1 - e0 + TP_ROWS - 1) / TP_ROWS;
  if (ntile > 0) stage(0, e0);
  if (ntile > 1) stage(1, e0 + TP_ROWS);
  for (int it = 0; it < ntile; ++it) {
    if (it + 1 < ntile) cp_async_wait<1>();
    else cp_async_wait<0>();
    __syncthreads();
    const float* vs = tsm + (size_t)(it & 1) * 2 * TP_ROWS * TP_LD;
    const float* ws = vs + TP_ROWS * TP_LD;
#pragma unroll 1
    for (int ks = 0; ks < 2; ++ks) {
      const int ea = warp * 16 + ks * 8 + t, eb = ea + 4;  // rows of the k8 step
      unsigned ahi[2][4], alo[2][4];
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        // real rows m = 16 mt + g (+ 8): word 16 mt + g (+ 8) of a staged row
        const int w0 = 16 * mt + g;
        tf32_split(vs[ea * TP_LD + w0], ahi[mt][0], alo[mt][0]);
        tf32_split(vs[ea * TP_LD + w0 + 8], ahi[mt][1], alo[mt][1]);
        tf32_split(vs[eb * TP_LD + w0], ahi[mt][2], alo[mt][2]);
        tf32_split(vs[eb * TP_LD + w0 + 8], ahi[mt][3], alo[mt][3]);
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        unsigned bh0, bl0, bh1, bl1;
        tf32_split(ws[ea * TP_LD + 8 * nt + g], bh0, bl0);
        tf32_split(ws[eb * TP_LD + 8 * nt + g], bh1, bl1);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
          mma_tf32(acc[mt][nt], alo[mt], bh0, bh1);
          mma_tf32(acc[mt][nt], ahi[mt], bl0, bl1);
          mma_tf32(acc[mt][nt], ahi[mt], bh0, bh1);
        }
      }
    }
    __syncthreads();
    if (it + 2 < ntile) stage(it & 1, e0 + (it + 2) * TP_ROWS);
  }
  // P tiles of the four warps into shared memory: warp w's P(m, n) at
  // red[w][m][n] (32 x 33 floats), d0 (m = 16 mt + g, n = 8 nt + 2t), d1 n + 1,
  // d2, d3 at m + 8
  float* red = tsm;
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const int m = 16 * mt + g, n = 8 * nt + 2 * t;
      float* rw = red + warp * 32 * 33;
      rw[m * 33 + n] = acc[mt][nt][0];
      rw[m * 33 + n + 1] = acc[mt][nt][1];
      rw[(m + 8) * 33 + n] = acc[mt][nt][2];
      rw[(m + 8) * 33 + n + 1] = acc[mt][nt][3];
    }
  __syncthreads();
  // thread -> 2 of the 256 complex outputs (i, j) of the tile
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int o = tid + 128 * h, li = o >> 4, lj = o & 15;
    if (ib + li >= K || lj >= r) continue;
    double pr = 0, pi = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const float* rw = red + w * 32 * 33;
      pr += (double)rw[(2 * li) * 33 + 2 * lj] + (double)rw[(2 * li + 1) * 33 + 2 * lj + 1];
      pi += (double)rw[(2 * li) * 33 + 2 * lj + 1] - (double)rw[(2 * li + 1) * 33 + 2 * lj];
    }
    part[((size_t)(blockIdx.z * nct + blockIdx.x) * kcap + ib + li) * BG_MAX + lj] = make_double2(pr, pi);
  }
}

// ------------------------------------------------------------ narrow blocks
// Blocks of few columns (few directions in a call: one plane wave is one
// column).  The tensor-core tiles are 16 columns wide, so these would multiply
// mostly zeros and split every basis value into TF32 parts for them; per basis
// value there are only 8 r FP32 operations, which the FP32 lanes do while the
// basis streams through at the rate of memory.  Same set, partial sums and
// results as the kernels above.  Up to BG_NARROW columns for the projection (its
// sums of 8 basis columns fill the registers beyond that), up to BG_NARROW_UPD
// for the update (at 16 the FP32 lanes would take as long as the tensor-core
// kernel, 6.6 ms of operations against its 7.6 at 256 x 256, 64 directions).
// Measured in a solve to 1e-10 on a GB300, tensor-core kernels and these:
//   1024 x 1024, 3 directions: projections 11.1 -> 4.0 ms, updates 10.9 -> 3.6
//   512 x 512, 8 directions:   updates 4.25 -> 2.93 ms
//   whole solve, 512 x 512, 1 direction 11.5 -> 7.5 ms; 256 x 256, 1 direction
//   5.0 -> 3.7 ms (pair operator 0.2 and 0.1 ms of it)
#define BG_NARROW 4
#define BG_NARROW_UPD 8

// update: one thread per two rows, the group's coefficients in shared memory
template <int RN>
__global__ void __launch_bounds__(256) k_bnn_narrow(BGSet set, const double2* __restrict__ cmat,
                                                    int nap, float beta, float sgn) {
  extern __shared__ float2 ncs[];   // [Kv][RN]
  const BGrp& gd = set.g[blockIdx.z];
  const int Kv = gd.Kv, r = gd.r, n = gd.n, tid = threadIdx.x;
  const int row0 = blockIdx.x * 512;
  if (row0 >= n) return;  // uniform over the block
  const double2* Cm = cmat + gd.coff;
  for (int i = tid; i < Kv * RN; i += 256) {
    const int q = i / RN, j = i % RN;
    const double2 c = j < r ? Cm[(size_t)q * BG_MAX + j] : make_double2(0.0, 0.0);
    ncs[i] = make_float2((float)(sgn * c.x), (float)(sgn * c.y));
  }
  __syncthreads();
  const int e0 = row0 + tid, e1 = e0 + 256;
  const float2* v0 = gd.V + min(e0, n - 1);
  const float2* v1 = gd.V + min(e1, n - 1);
  float2 a0[RN], a1[RN];
#pragma unroll
  for (int j = 0; j < RN; ++j) a0[j] = a1[j] = make_float2(0.f, 0.f);
  auto add = [&](float2 x, float2 y, const float2* c) {
#pragma unroll
    for (int j = 0; j < RN; ++j) {
      const float2 w = c[j];
      a0[j].x = fmaf(x.x, w.x, fmaf(-x.y, w.y, a0[j].x));
      a0[j].y = fmaf(x.x, w.y, fmaf(x.y, w.x, a0[j].y));
      a1[j].x = fmaf(y.x, w.x, fmaf(-y.y, w.y, a1[j].x));
      a1[j].y = fmaf(y.x, w.y, fmaf(y.y, w.x, a1[j].y));
    }
  };
  int i = 0;
  for (; i + 8 <= Kv; i += 8) {
    float2 x[8], y[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      x[u] = v0[(size_t)(i + u) * nap];
      y[u] = v1[(size_t)(i + u) * nap];
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) add(x[u], y[u], ncs + (i + u) * RN);
  }
  for (; i < Kv; ++i) add(v0[(size_t)i * nap], v1[(size_t)i * nap], ncs + i * RN);
#pragma unroll
  for (int j = 0; j < RN; ++j) {
    if (j >= r) break;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = h ? e1 : e0;
      if (e >= n) break;
      const float2 s = h ? a1[j] : a0[j];
      const float2 o = beta != 0.f ? gd.W[(size_t)j * nap + e] : make_float2(0.f, 0.f);
      gd.O[(size_t)j * nap + e] = make_float2(fmaf(beta, o.x, s.x), fmaf(beta, o.y, s.y));
    }
  }
}

// projection: a block takes NP_KC basis columns against all block columns over
// its slab, each thread its rows in FP32; the threads' sums are added by a
// halving exchange within the warp, the warps' in FP64
#define NP_KC 8
template <int RN>
__global__ void __launch_bounds__(128, 4) k_bproj_narrow(BGSet set, double2* __restrict__ part,
                                                         int nap, int rs, int nct, int kcap) {
  constexpr int NV = NP_KC * RN * 2;
  __shared__ float red[4][NV];
  const BGrp& gd = set.g[blockIdx.z];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ib = blockIdx.y * NP_KC, K = gd.K, Kv = gd.Kv, r = gd.r;
  if (ib >= K) return;  // uniform over the block
  const int e0 = blockIdx.x * rs, e1 = min(gd.n, e0 + rs);
  const float2* src[NP_KC];
#pragma unroll
  for (int u = 0; u < NP_KC; ++u) {
    const int i = min(ib + u, K - 1);
    src[u] = i < Kv ? gd.V + (size_t)i * nap : gd.W + (size_t)(i - Kv) * nap;
  }
  float acc[NV];   // [u][j][re, im]
#pragma unroll
  for (int q = 0; q < NV; ++q) acc[q] = 0.f;
  for (int e = e0 + tid; e < e1; e += 128) {
    float2 x[NP_KC], w[RN];
#pragma unroll
    for (int u = 0; u < NP_KC; ++u) x[u] = __ldg(src[u] + e);
#pragma unroll
    for (int j = 0; j < RN; ++j) w[j] = __ldg(gd.W + (size_t)min(j, r - 1) * nap + e);
#pragma unroll
    for (int u = 0; u < NP_KC; ++u)
#pragma unroll
      for (int j = 0; j < RN; ++j) {   // conj(x) w
        float* a = acc + (u * RN + j) * 2;
        a[0] = fmaf(x[u].x, w[j].x, fmaf(x[u].y, w[j].y, a[0]));
        a[1] = fmaf(x[u].x, w[j].y, fmaf(-x[u].y, w[j].x, a[1]));
      }
  }
  // lane exchange: while the count is even, a lane keeps one half of the sums
  int base = 0;
  auto step = [&](auto cnt, int o) {
    constexpr int H = decltype(cnt)::value / 2;
    const bool up = lane & o;
#pragma unroll
    for (int k = 0; k < H; ++k) {
      const float keep = up ? acc[k + H] : acc[k], send = up ? acc[k] : acc[k + H];
      acc[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
    base += up ? H : 0;
  };
  step(std::integral_constant<int, NV>{}, 16);
  step(std::integral_constant<int, NV / 2>{}, 8);
  step(std::integral_constant<int, NV / 4>{}, 4);
  step(std::integral_constant<int, NV / 8>{}, 2);
  constexpr int L = NV / 16;   // RN sums are left
#pragma unroll
  for (int k = 0; k < L; ++k) {
    acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], 1);
    if (!(lane & 1)) red[warp][base + k] = acc[k];
  }
  __syncthreads();
  for (int q = tid; q < NP_KC * RN; q += 128) {
    const int u = q / RN, j = q % RN;
    if (ib + u >= K || j >= r) continue;
    double pr = 0, pi = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      pr += (double)red[w][2 * q];
      pi += (double)red[w][2 * q + 1];
    }
    part[((size_t)(blockIdx.z * nct + blockIdx.x) * kcap + ib + u) * BG_MAX + j] = make_double2(pr, pi);
  }
}

// dst[map[c]] += src[c]  (column c of a contiguous block; grid (ceil(nap/256), ncol))
__global__ void k_scatter_add(const float2* __restrict__ src, float2* __restrict__ dst,
                              const int* __restrict__ map, int nap) {
  const int c = blockIdx.y, e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nap) return;
  const float2 a = src[(size_t)c * nap + e];
  float2* o = dst + (size_t)map[c] * nap + e;
  *o = make_float2(o->x + a.x, o->y + a.y);
}

// dst[c] = src[map[c]], from the order of Appendix A into that of pm (gather
// into a contiguous block); one thread per mode pair (m, n), grid
// (ceil(nx ny / 256), ncol)
__global__ void k_gather_cols(const float2* __restrict__ src, float2* __restrict__ dst,
                              const int* __restrict__ map, int nap, int nx, int ny, int n1, int n2,
                              ParityMap pm) {
  const int c = blockIdx.y, i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nx * ny) return;
  const int m = i / ny, n = i - m * ny, N = ny - 1;
  const float2* s = src + (size_t)map[c] * nap;
  float2* d = dst + (size_t)c * nap;
  const int i1 = m * N + (n - 1), i2 = n1 + (m - 1) * ny + n, i3 = n1 + n2 + (m - 1) * N + (n - 1);
  if (n >= 1) d[pm.on ? pm.e1(m, n) : i1] = s[i1];
  if (m >= 1) d[pm.on ? pm.e2(m, n) : i2] = s[i2];
  if (m >= 1 && n >= 1) d[pm.on ? pm.e3(m, n) : i3] = s[i3];
}

// dst[c] -= src[c]  (contiguous blocks; grid (ceil(nap/256), ncol))
__global__ void k_sub_cols(const float2* __restrict__ src, float2* __restrict__ dst, int nap) {
  const size_t k = (size_t)blockIdx.y * nap + blockIdx.x * blockDim.x + threadIdx.x;
  if (blockIdx.x * blockDim.x + threadIdx.x >= (unsigned)nap) return;
  dst[k] = make_float2(dst[k].x - src[k].x, dst[k].y - src[k].y);
}

static inline unsigned bg_blocks(long long n, int b) { return (unsigned)((n + b - 1) / b); }

// ------------------------------------------------------------------ host side
// (herm_eig, cholqr, svqb, matmul_left, BlockLS: bgmres_host.h)

struct BWork {
  float2 *V, *Rc, *Z, *Wb, *Tt;
  double2 *part, *hb, *cb;
  int* map;
  void* apw;
  int vcap;         // basis columns of a group
  int kcap, emax;   // rows of a system's coefficients, systems
};

static size_t al256(size_t x) { return (x + 255) / 256 * 256; }

// Directions per group: the option where it was set, else 16, or 8 on small
// grids: the host's least squares take time proportional to the square of the
// width, and below 30,000 unknowns a block step on the GPU is shorter than
// they are at 16 (64 x 64, 64 directions: 8.5 ms a solve at 16, 7.1 ms at 8).
static int group_width(const cavity_ctx* ctx) {
  const int o = std::max(1, std::min(BG_MAX, ctx->opt[CAVITY_OPT_GROUP_WIDTH]));
  if (ctx->gw_set) return o;
  return ctx->g.nap < 30000 ? std::min(o, 8) : o;
}
// Parity classes (see run_block_inner) where they pay: the operator steps they
// save must be worth their coefficients and the second Gram-Schmidt pass they
// need.  Measured, one solve to 1e-10 with one and with four classes: 256 x 256,
// 64 directions (196,000 unknowns) 73 and 78 ms; 512 x 512, 8 directions
// (784,000) 48.5 and 44.3 ms; 1024 x 1024, 3 directions 163 and 103 ms.  Not
// with the coarse level of the preconditioner, a solve in the order of
// Appendix A.
#define BG_CLASS_ROWS 300000
static int num_classes(const cavity_ctx* ctx) {
  return ctx->opt[CAVITY_OPT_COARSE_MODES] > 0 || ctx->g.nap < BG_CLASS_ROWS ? 1 : BG_CLASSES;
}

// work area of a call for up to ndir directions (it takes up to BG_GROUPS
// groups at a time), V .. cb per group and class
struct BSizes {
  int nd, gm, em;   // directions, groups, systems
  size_t vcap;      // basis columns of a group: as wide as its block may be
  size_t kcap, col;
  BSizes(const cavity_ctx* ctx, int ndir, int mb) {
    const int gw = group_width(ctx);
    nd = std::min(ndir, BG_GROUPS * gw);
    gm = (nd + gw - 1) / gw;
    em = gm * num_classes(ctx);
    vcap = (size_t)(mb + 1) * gw;
    kcap = (size_t)(mb + 1) * BG_MAX;
    col = sizeof(float2) * (size_t)ctx->g.nap;
  }
};
size_t block_inner_work_bytes(const cavity_ctx* ctx, int ndir, int mb) {
  const BSizes z(ctx, ndir, mb);
  size_t b = 0;
  b += al256(z.col * z.gm * z.vcap);                              // V
  b += 4 * al256(z.col * z.nd);                                   // Rc, Z, Wb, Tt
  b += al256(sizeof(double2) * BG_PART_CTAS * z.kcap * BG_MAX);   // part
  b += al256(sizeof(double2) * 3 * z.em * z.kcap * BG_MAX);       // hb
  b += al256(sizeof(double2) * z.em * z.kcap * BG_MAX);           // cb
  b += al256(sizeof(int) * z.nd);                                 // map
  b += al256(apply_work_bytes(ctx->g, z.nd, sizeof(float2)));
  return b;
}

static BWork bwork_carve(void* base, const cavity_ctx* ctx, int ndir, int mb) {
  const BSizes z(ctx, ndir, mb);
  char* p = (char*)base;
  BWork w;
  w.V = (float2*)p; p += al256(z.col * z.gm * z.vcap);
  w.Rc = (float2*)p; p += al256(z.col * z.nd);
  w.Z = (float2*)p; p += al256(z.col * z.nd);
  w.Wb = (float2*)p; p += al256(z.col * z.nd);
  w.Tt = (float2*)p; p += al256(z.col * z.nd);
  w.part = (double2*)p; p += al256(sizeof(double2) * BG_PART_CTAS * z.kcap * BG_MAX);
  w.hb = (double2*)p; p += al256(sizeof(double2) * 3 * z.em * z.kcap * BG_MAX);
  w.cb = (double2*)p; p += al256(sizeof(double2) * z.em * z.kcap * BG_MAX);
  w.map = (int*)p; p += al256(sizeof(int) * z.nd);
  w.apw = p;
  w.vcap = (int)z.vcap;
  w.kcap = (int)z.kcap;
  w.emax = z.em;
  return w;
}

static int max_rows(const BGSet& set, int ng) {
  int n = 0;
  for (int t = 0; t < ng; ++t) n = std::max(n, set.g[t].n);
  return n;
}

static int max_r(const BGSet& set, int ng) {
  int r = 0;
  for (int t = 0; t < ng; ++t) r = std::max(r, set.g[t].r);
  return r;
}
// f(RN) with RN >= r a compile-time constant, 1 <= r <= MOST (4 or 8)
template <int MOST, typename F> static void narrow_dispatch(int r, F f) {
  if (r == 1) f(std::integral_constant<int, 1>{});
  else if (r == 2) f(std::integral_constant<int, 2>{});
  else if (r == 3) f(std::integral_constant<int, 3>{});
  else if (MOST == 4 || r == 4) f(std::integral_constant<int, 4>{});
  else if constexpr (MOST == 8) {
    if (r <= 6) f(std::integral_constant<int, 6>{});
    else f(std::integral_constant<int, 8>{});
  }
}

// V^H W for every system of `set` (ng of them, K and r each) into
// hb + slot * emax * kcap * BG_MAX, laid out [z][i][j].
static void bproj(cavity_ctx* ctx, const BGSet& set, int ng, int kmax, const BWork& w, int slot) {
  const int nap = ctx->g.nap, nrow = max_rows(set, ng);
  const int rm = max_r(set, ng);
  const bool narrow = rm <= BG_NARROW;
  const int ytiles = narrow ? (kmax + NP_KC - 1) / NP_KC : (kmax + 15) / 16;
  // slabs of rows such that slabs x column tiles x groups fill one wave of
  // resident blocks (four per SM, BG_PART_CTAS in all): no tail wave, and a
  // short projection (the Gram matrix, K = 16) still spreads over every SM
  int nct = std::max(1, BG_PART_CTAS / (ytiles * ng));
  nct = std::min(nct, (nrow + BP_ROWS - 1) / BP_ROWS);
  int rs = (nrow + nct - 1) / nct;
  rs = (rs + BP_ROWS - 1) / BP_ROWS * BP_ROWS;
  nct = (nrow + rs - 1) / rs;
  double2* h = w.hb + (size_t)slot * w.emax * w.kcap * BG_MAX;
  static DeviceFlag done;
  if (!done) {
    cudaFuncSetAttribute(k_bproj_tc<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TP_SMEM);
    cudaFuncSetAttribute(k_bproj_tc<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TP_SMEM);
    done.set();
  }
  if (narrow) {
    KScope ks_(ctx, KC_KRYLOV);
    narrow_dispatch<BG_NARROW>(rm, [&](auto c) {
      k_bproj_narrow<decltype(c)::value><<<dim3(nct, ytiles, ng), 128, 0, ctx->stream>>>(
          set, w.part, nap, rs, nct, w.kcap);
    });
  } else {
    KScope ks_(ctx, KC_KRYLOV);
    if (rm <= 8)
      k_bproj_tc<2><<<dim3(nct, ytiles, ng), 128, TP_SMEM, ctx->stream>>>(set, w.part, nap, rs, nct,
                                                                          w.kcap);
    else
      k_bproj_tc<4><<<dim3(nct, ytiles, ng), 128, TP_SMEM, ctx->stream>>>(set, w.part, nap, rs, nct,
                                                                          w.kcap);
  }
  {
    KScope ks_(ctx, KC_KRYLOV);
    k_bproj_final<<<dim3(kmax, ng), 256, 0, ctx->stream>>>(set, w.part, h, nct, w.kcap);
  }
}

static cavity_status bnn(cavity_ctx* ctx, const BGSet& set, int ng, const double2* cmat, float beta,
                         float sgn) {
  const int nap = ctx->g.nap;
  KScope ks_(ctx, KC_KRYLOV);
  const int rm = max_r(set, ng);
  if (rm <= BG_NARROW_UPD) {
    int kv = 0;
    for (int t = 0; t < ng; ++t) kv = std::max(kv, set.g[t].Kv);
    narrow_dispatch<BG_NARROW_UPD>(rm, [&](auto c) {
      constexpr int RN = decltype(c)::value;
      k_bnn_narrow<RN><<<dim3(bg_blocks(max_rows(set, ng), 512), 1, ng), 256,
                         sizeof(float2) * RN * kv, ctx->stream>>>(set, cmat, nap, beta, sgn);
    });
    return CAVITY_OK;
  }
  k_bnn_tc5<<<dim3(bg_blocks(max_rows(set, ng), 128), 1, ng), 128, 2 * sizeof(T5Buf), ctx->stream>>>(
      set, cmat, nap, beta, sgn);
  return CAVITY_OK;
}

// Solves A M^{-1} y = r_d for the directions with active[d] (r: ndir scaled
// FP32 residual columns), accumulating d = M^{-1} y into the d columns (zeroed
// first).  tol[d] is the relative target (the columns have unit norm); iters[d]
// is increased by the block steps taken, est[d] is the final least-squares
// residual.  Groups still above tolerance after mb steps restart from their
// true inner residual.
//
// Parity classes.  A couples only modes of one parity class, so each class of
// a group has its own basis (the rows of its class in the group's columns), its
// own coefficients and its own least-squares problem, while one application of
// the operator to the columns serves all four.  Every class then minimises its
// own residual over its own block space: fewer steps for the same operator
// work (512 x 512, 8 directions: 19 block steps to 1e-10 against 22; 1024 x
// 1024, 3 directions: 22 against 39), and a pass of the orthogonalisation does
// the same number of operations.
// Systems are numbered e = z NC + c (group z, class c).
cavity_status run_block_inner(cavity_ctx* ctx, int ndir, const float2* r, float2* d,
                              const std::vector<double>& tol, const std::vector<char>& active, int mb,
                              int maxit, void* work, std::vector<int>& iters,
                              std::vector<double>& est) {
  const Geo& g = ctx->g;
  const int nap = g.nap;
  cudaStream_t st = ctx->stream;
  CK(cudaMemsetAsync(d, 0, sizeof(float2) * (size_t)ndir * nap, st));
  std::vector<int> all;
  for (int q = 0; q < ndir; ++q)
    if (active[q]) all.push_back(q);
  est.assign(ndir, 0.0);
  const int NC = num_classes(ctx);
  const ParityMap pm = NC > 1 ? parity_map(g) : ParityMap();
  auto crow = [&](int c) { return NC > 1 ? pm.base[c] : 0; };
  auto clen = [&](int c) { return NC > 1 ? pm.base[c + 1] - pm.base[c] : nap; };
  // directions beyond one call's capacity are solved in further batches
  const int gw = group_width(ctx);
  for (size_t b0 = 0; b0 < all.size(); b0 += (size_t)BG_GROUPS * gw) {
    const int na = (int)std::min(all.size() - b0, (size_t)BG_GROUPS * gw);
    std::vector<int> dirs(all.begin() + b0, all.begin() + b0 + na);
    BWork w = bwork_carve(work, ctx, ndir, mb);
    const int ng = (na + gw - 1) / gw, ne = ng * NC;
    // balanced groups: group z holds directions [goff[z], goff[z] + gr[z])
    std::vector<int> gr(ng), goff(ng);
    for (int z = 0, o = 0; z < ng; ++z) {
      gr[z] = na / ng + (z < na % ng ? 1 : 0);
      goff[z] = o;
      o += gr[z];
    }
    auto er = [&](int e) { return gr[e / NC]; };
    CK(cudaMemcpyAsync(w.map, dirs.data(), sizeof(int) * na, cudaMemcpyHostToDevice, st));
    {
      KScope ks_(ctx, KC_KRYLOV);
      k_gather_cols<<<dim3(bg_blocks((long long)g.nx * g.ny, 256), na), 256, 0, st>>>(
          r, w.Rc, w.map, nap, g.nx, g.ny, g.n1, g.n2, pm);
    }
    std::vector<char> gdone(ng, 0);
    int used = 0;
    auto Vg = [&](int z) { return w.V + (size_t)z * w.vcap * nap; };
    // column col of system e's basis, at its class' rows
    auto Ve = [&](int e, int col) { return Vg(e / NC) + (size_t)col * nap + crow(e % NC); };
    auto hptr = [&](int slot, int e) {
      return w.hb + ((size_t)slot * w.emax + e) * w.kcap * BG_MAX;
    };
    const size_t hsz = (size_t)w.kcap * BG_MAX;
    // pinned staging: three fetched coefficient slots, then the upload slot;
    // an upload is rewritten only after a stream synchronisation that follows
    // the previous one
    CKS(ensure_pin(ctx, sizeof(double2) * 4 * w.emax * hsz));
    double2* hh = (double2*)ctx->pin;
    double2* cup = hh + (size_t)3 * w.emax * hsz;
    bool upl_pending = false;  // an upload may still be queued behind GPU work
    auto sync = [&]() -> cavity_status {
      CK(cudaStreamSynchronize(st));
      upl_pending = false;
      return CAVITY_OK;
    };
    // the first `rows` rows of n systems' coefficients in a slot
    auto fetch = [&](int slot, int n, int rows) -> cavity_status {
      CK(cudaMemcpy2DAsync(hh + (size_t)slot * w.emax * hsz, sizeof(double2) * hsz, hptr(slot, 0),
                           sizeof(double2) * hsz, sizeof(double2) * rows * BG_MAX, n,
                           cudaMemcpyDeviceToHost, st));
      return CAVITY_OK;
    };
    auto hval = [&](int slot, int t, int i, int j) {
      const double2 v = hh[((size_t)slot * w.emax + t) * hsz + (size_t)i * BG_MAX + j];
      return cd(v.x, v.y);
    };
    // matrix t of mats into coefficient slot t of the device
    auto upload = [&](const std::vector<std::vector<cd>>& mats) -> cavity_status {
      if (upl_pending) CKS(sync());
      size_t most = 0;
      for (size_t q = 0; q < mats.size(); ++q) {
        const auto& m = mats[q];
        most = std::max(most, m.size());
        for (size_t t = 0; t < m.size(); ++t)
          cup[q * hsz + t] = make_double2(m[t].real(), m[t].imag());
      }
      CK(cudaMemcpy2DAsync(w.cb, sizeof(double2) * hsz, cup, sizeof(double2) * hsz,
                           sizeof(double2) * most, mats.size(), cudaMemcpyHostToDevice, st));
      upl_pending = true;
      return CAVITY_OK;
    };
    // Orthonormalise block columns [col0, col0 + r) of each listed system's
    // basis in place by repeated SVQB; S[q] receives the r x r factor with
    // old block = new block * S, amp[q] how far its transforms magnify a column
    // (root mean square of T's column norms, 1 for an orthonormal block; the
    // largest norm instead left the block steps of 55 of 57 solves on grids of
    // 300,000 unknowns and more as they are, repeated and nearly equal directions
    // among them, and moved two by one).  G0, when given, holds the Gram
    // matrices of the blocks as they are (first pass without a device Gram).
    auto orthonormalise = [&](const std::vector<int>& es, const std::vector<int>& col0,
                              std::vector<std::vector<cd>>& S, std::vector<double>& amp,
                              const std::vector<std::vector<cd>>* G0) -> cavity_status {
      const int nz = (int)es.size();
      S.assign(nz, {});
      amp.assign(nz, 1.0);
      std::vector<char> ok(nz, 0);
      for (int pass = 0; pass < 4; ++pass) {
        std::vector<int> todo;
        for (int q = 0; q < nz; ++q)
          if (!ok[q]) todo.push_back(q);
        if (todo.empty()) break;
        if (pass > 0 || !G0) {
          BGSet set;
          for (size_t t = 0; t < todo.size(); ++t) {
            const int q = todo[t], e = es[q];
            float2* blk = Ve(e, col0[q]);
            set.g[t] = BGrp{blk, blk, blk, clen(e % NC), 0, er(e), er(e), 0};
          }
          bproj(ctx, set, (int)todo.size(), BG_MAX, w, 2);
          CKS(fetch(2, (int)todo.size(), BG_MAX));
          CKS(sync());
        }
        std::vector<std::vector<cd>> Ts;
        BGSet set2;
        int n2 = 0;
        for (size_t t = 0; t < todo.size(); ++t) {
          const int q = todo[t], e = es[q], n = er(e);
          std::vector<cd> G((size_t)n * n);
          if (pass == 0 && G0) G = (*G0)[q];
          else
            for (int i = 0; i < n; ++i)
              for (int j = 0; j < n; ++j) G[(size_t)i * n + j] = hval(2, (int)t, i, j);
          double dev = 0;
          for (int i = 0; i < n; ++i)
            for (int j = 0; j < n; ++j)
              dev = std::max(dev, std::abs(G[(size_t)i * n + j] - (i == j ? 1.0 : 0.0)));
          if (pass > 0 && dev <= 2e-6) {
            ok[q] = 1;
            continue;
          }
          // Cholesky QR; its FP32 transform leaves an orthogonality error
          // within the block of ~ eps32 cond(G), accepted without a check for
          // cond(G) <= 1e3: it perturbs the least-squares residual norms by
          // that relative amount, far below the inner tolerance, while the
          // orthogonality to the earlier blocks comes from the Gram-Schmidt pass
          // before (and, with parity classes, the second one below).  Nearly
          // dependent blocks take the eigendecomposition and further passes.
          std::vector<cd> T, Sk;
          double cond = 1e300, ratio;
          if (cholqr(G, n, T, Sk, cond)) {
            if (cond <= 1e3) ok[q] = 1;
          } else {
            svqb(G, n, T, Sk, ratio);
          }
          if (S[q].empty()) S[q] = Sk;
          else matmul_left(Sk, S[q], n);
          double tn = 0;
          for (const cd& x : T) tn += std::norm(x);
          amp[q] *= std::sqrt(tn / n);
          Ts.push_back(T);
          float2* blk = Ve(e, col0[q]);
          set2.g[n2] = BGrp{blk, blk, blk, clen(e % NC), n, n, n, n2 * (int)hsz};
          ++n2;
        }
        if (n2 == 0) break;
        CKS(upload(Ts));
        CKS(bnn(ctx, set2, n2, w.cb, 0.f, 1.f));
      }
      for (int q = 0; q < nz; ++q)
        if (S[q].empty()) {  // first pass always transforms, so this is unreachable
          const int n = er(es[q]);
          S[q].assign((size_t)n * n, cd(0, 0));
          for (int i = 0; i < n; ++i) S[q][(size_t)i * n + i] = 1.0;
        }
      return CAVITY_OK;
    };

    while (true) {
      std::vector<int> cyc;   // groups of this cycle
      for (int z = 0; z < ng; ++z)
        if (!gdone[z]) cyc.push_back(z);
      if (cyc.empty() || used >= maxit) break;
      // cycle start: V_0 = orthonormalised residual block of each system
      std::vector<int> run;   // systems of the step being processed, in slot order
      for (int z : cyc) {
        CK(cudaMemcpyAsync(Vg(z), w.Rc + (size_t)goff[z] * nap, sizeof(float2) * gr[z] * nap,
                           cudaMemcpyDeviceToDevice, st));
        for (int c = 0; c < NC; ++c) run.push_back(z * NC + c);
      }
      std::vector<std::vector<cd>> S0;
      std::vector<double> amp;
      CKS(orthonormalise(run, std::vector<int>(run.size(), 0), S0, amp, nullptr));
      std::vector<BlockLS> ls(ne);
      for (size_t q = 0; q < run.size(); ++q) ls[run[q]].start(er(run[q]), S0[q]);
      std::vector<char> cdone(ng, 0), edone(ne, 0);
      // a system is done with its group, or when none of its directions has
      // more than a quarter of its tolerance left (four classes then stay
      // below half of it together)
      auto settle = [&](int e) {
        const int z = e / NC;
        bool low = true;
        for (int j = 0; j < gr[z]; ++j) low = low && ls[e].resid(j) <= 0.25 * tol[dirs[goff[z] + j]];
        if (low && NC > 1) edone[e] = 1;
      };
      for (int e : run) settle(e);
      auto running = [&](const std::vector<int>& from) {
        std::vector<int> out;
        for (int e : from)
          if (!edone[e] && !cdone[e / NC]) out.push_back(e);
        return out;
      };
      // GPU work of block step k for the systems in `es`: W = A M^{-1} V_k of
      // their groups' columns, one classical Gram-Schmidt pass into basis slot
      // k + 1, the Gram matrix of the result, and the coefficients on their way
      // to the host
      std::vector<int> woff(ng, 0);
      auto launch_step = [&](int k, const std::vector<int>& es) -> cavity_status {
        std::vector<char> in(ne, 0);
        for (int e : es) in[e] = 1;
        std::vector<int> zs;
        for (int e : es)
          if (zs.empty() || zs.back() != e / NC) zs.push_back(e / NC);
        // rows of classes that are done (not written by the last step): zero, so
        // that nothing of them is in the columns the operator takes
        for (int z : zs)
          for (int c = 0; c < NC; ++c)
            if (!in[z * NC + c])
              CK(cudaMemset2DAsync(Ve(z * NC + c, k * gr[z]), sizeof(float2) * nap, 0,
                                   sizeof(float2) * clen(c), gr[z], st));
        int nc = 0;
        PcCols cols;
        for (int z : zs) {
          woff[z] = nc;
          cols.first[cols.n] = nc;
          cols.src[cols.n++] = Vg(z) + (size_t)k * gr[z] * nap;
          nc += gr[z];
        }
        CKS(launch_precond_groups(ctx, nc, cols, w.Z, pm));
        CKS(launch_apply<float>(ctx, nc, w.Z, w.Wb, w.apw, nap, pm));
        BGSet set, gs;
        int kmax = 0;
        for (size_t t = 0; t < es.size(); ++t) {
          const int e = es[t], kv = (k + 1) * er(e), n = clen(e % NC);
          float2* we = w.Wb + (size_t)woff[e / NC] * nap + crow(e % NC);
          float2* vn = Ve(e, kv);   // the projected block goes straight into its basis slot
          set.g[t] = BGrp{Ve(e, 0), we, vn, n, kv, kv, er(e), (int)(t * hsz)};
          // Gram matrix of the projected block, formed from it directly (the
          // difference G(W) - H^H H cancels when W lies almost in the basis)
          gs.g[t] = BGrp{vn, vn, vn, n, 0, er(e), er(e), 0};
          kmax = std::max(kmax, kv);
        }
        const int nr = (int)es.size();
        bproj(ctx, set, nr, kmax, w, 0);
        CKS(bnn(ctx, set, nr, hptr(0, 0), 1.f, -1.f));
        bproj(ctx, gs, nr, BG_MAX, w, 1);
        CKS(fetch(0, nr, kmax));
        CKS(fetch(1, nr, BG_MAX));
        return CAVITY_OK;
      };
      // residual estimates of the last two steps per direction (convergence
      // forecast for launching the next step before the least squares)
      std::vector<double> e1(ndir, 1.0), e2(ndir, 1.0);
      // estimates of a group from its systems; marks it when all are below
      // tolerance
      auto estimate = [&](int z) {
        bool conv = true;
        for (int j = 0; j < gr[z]; ++j) {
          const int dd = dirs[goff[z] + j];
          double s = 0;
          for (int c = 0; c < NC; ++c) {
            const double v = ls[z * NC + c].resid(j);
            s += v * v;
          }
          est[dd] = std::sqrt(s);
          e2[dd] = e1[dd];
          e1[dd] = est[dd];
          conv = conv && est[dd] <= tol[dd];
        }
        if (conv) cdone[z] = 1;
      };
      for (int z : cyc) estimate(z);
      // run: the systems of the step being processed, in launch (slot) order;
      // a system that finished under a step launched ahead stays in it but
      // takes no further least-squares columns
      run = running(run);
      std::vector<int> lnext;
      bool launched = false;
      int k = 0;
      for (; k < mb && used < maxit; ++k) {
        if (run.empty()) break;
        if (!launched) CKS(launch_step(k, run));
        launched = false;
        CKS(sync());
        // Gram matrix of the projected block (slot 1)
        std::vector<std::vector<cd>> G0(run.size()), Hc(run.size());
        for (size_t t = 0; t < run.size(); ++t) {
          const int n = er(run[t]), K = (k + 1) * n;
          auto& G = G0[t];
          G.assign((size_t)n * n, cd(0, 0));
          for (int i = 0; i < n; ++i)
            for (int j = 0; j < n; ++j) G[(size_t)i * n + j] = hval(1, (int)t, i, j);
          for (int i = 0; i < n; ++i)  // exactly Hermitian
            for (int j = 0; j < i; ++j) {
              const cd m = 0.5 * (G[(size_t)i * n + j] + std::conj(G[(size_t)j * n + i]));
              G[(size_t)i * n + j] = m;
              G[(size_t)j * n + i] = std::conj(m);
            }
          Hc[t].resize((size_t)K * n);  // H, kept before the slots are reused
          for (int i = 0; i < K; ++i)
            for (int j = 0; j < n; ++j) Hc[t][(size_t)i * n + j] = hval(0, (int)t, i, j);
        }
        std::vector<std::vector<cd>> S;
        std::vector<int> c0;
        for (int e : run) c0.push_back((k + 1) * er(e));
        CKS(orthonormalise(run, c0, S, amp, &G0));
        // Second Gram-Schmidt pass where the transform magnified the rounding of
        // the first (2^-24 of the block before projection, which is not
        // orthogonal to the basis) by more than BG_REORTH: near convergence the
        // projected block of a class shrinks, and what orthogonality one pass
        // loses grows with the square of the residual reduction.  V' -= V (V^H V')
        // changes V' by about 2^-24 times the magnification, so V' stays
        // orthonormal and H as it is to rounding; beyond BG_REORTH_FULL (a nearly
        // dependent block) it is orthonormalised again and H corrected.
        std::vector<int> quick, full;   // indices into run
        for (size_t t = 0; t < run.size(); ++t) {
          if (NC == 1 || edone[run[t]] || cdone[run[t] / NC]) continue;
          const int n = er(run[t]), K = (k + 1) * n;
          double w0 = 0;
          for (int j = 0; j < n; ++j) {
            double q = G0[t][(size_t)j * n + j].real();
            for (int i = 0; i < K; ++i) q += std::norm(Hc[t][(size_t)i * n + j]);
            w0 = std::max(w0, q);
          }
          const double mag = amp[t] * std::sqrt(w0);
          if (mag > BG_REORTH_FULL) full.push_back((int)t);
          else if (mag > BG_REORTH) quick.push_back((int)t);
        }
        auto again = [&](const std::vector<int>& ts) -> cavity_status {
          BGSet set;
          int kmax = 0;
          for (size_t q = 0; q < ts.size(); ++q) {
            const int e = run[ts[q]], kv = c0[ts[q]];
            float2* vn = Ve(e, kv);
            set.g[q] = BGrp{Ve(e, 0), vn, vn, clen(e % NC), kv, kv, er(e), (int)(q * hsz)};
            kmax = std::max(kmax, kv);
          }
          bproj(ctx, set, (int)ts.size(), kmax, w, 0);
          return bnn(ctx, set, (int)ts.size(), hptr(0, 0), 1.f, -1.f);
        };
        if (!quick.empty()) CKS(again(quick));
        if (!full.empty()) {
          CKS(again(full));
          std::vector<int> es, ec;
          for (int t : full) {
            es.push_back(run[t]);
            ec.push_back(c0[t]);
          }
          CKS(fetch(0, (int)full.size(), (k + 1) * BG_MAX));
          std::vector<std::vector<cd>> S2;
          std::vector<double> amp2;
          CKS(orthonormalise(es, ec, S2, amp2, nullptr));   // synchronises: slot 0 is here
          for (size_t q = 0; q < full.size(); ++q) {
            const int t = full[q], n = er(run[t]), K = (k + 1) * n;
            // W = V' S with V' = V'' S2 + V H2:  H += H2 S, S <- S2 S
            for (int i = 0; i < K; ++i)
              for (int j = 0; j < n; ++j) {
                cd x = 0;
                for (int l = 0; l < n; ++l) x += hval(0, (int)q, i, l) * S[t][(size_t)l * n + j];
                Hc[t][(size_t)i * n + j] += x;
              }
            matmul_left(S2[q], S[t], n);
          }
        }
        ++used;
        // launch step k + 1 now unless some group is forecast to converge at
        // step k (geometric extrapolation of its estimates)
        const std::vector<int> ahead = running(run);
        bool soon = false;
        for (int z : cyc) {
          if (cdone[z]) continue;
          for (int j = 0; j < gr[z]; ++j) {
            const int dd = dirs[goff[z] + j];
            const double f = e2[dd] > 0 ? e1[dd] * std::min(1.0, e1[dd] / e2[dd]) : e1[dd];
            soon = soon || f <= 2.0 * tol[dd];
          }
        }
        if (!soon && k + 1 < mb && used < maxit) {
          CKS(launch_step(k + 1, ahead));
          launched = true;
          lnext = ahead;
        }
        // least squares of step k (overlaps the GPU work just launched)
        std::vector<char> stepped(ng, 0);
        for (size_t t = 0; t < run.size(); ++t) {
          const int e = run[t], z = e / NC, n = gr[z], K = (k + 1) * n;
          if (edone[e] || cdone[z]) continue;
          std::vector<std::vector<cd>> cols(n, std::vector<cd>((size_t)K + n, cd(0, 0)));
          for (int j = 0; j < n; ++j) {
            for (int i = 0; i < K; ++i) cols[j][i] = Hc[t][(size_t)i * n + j];
            for (int i = 0; i < n; ++i) cols[j][K + i] = S[t][(size_t)i * n + j];
          }
          ls[e].add(cols, K + n);
          settle(e);
          stepped[z] = 1;
        }
        for (int z : cyc) {
          if (!stepped[z]) continue;
          for (int j = 0; j < gr[z]; ++j) iters[dirs[goff[z] + j]] += 1;
          estimate(z);
        }
        const std::vector<int> next = running(run);
        if (next.empty()) break;
        run = launched ? lnext : next;
      }
      // corrections of this cycle: d += M^{-1} V Y per system (a system whose
      // residual vanished from the start has no columns: T = 0)
      std::vector<std::vector<cd>> Ys;
      BGSet set;
      int n = 0;
      for (int z : cyc)
        for (int c = 0; c < NC; ++c) {
          const int e = z * NC + c;
          std::vector<cd> Y;
          ls[e].solve(Y);
          set.g[n] = BGrp{Ve(e, 0), nullptr, w.Tt + (size_t)goff[z] * nap + crow(c), clen(c),
                          ls[e].cols, ls[e].cols, gr[z], n * (int)hsz};
          Ys.push_back(Y);
          ++n;
        }
      bool any = false;
      for (const auto& Y : Ys) any = any || !Y.empty();
      if (any) CKS(upload(Ys));
      CKS(bnn(ctx, set, n, w.cb, 0.f, 1.f));
      // T -> Z = M^{-1} T, scattered into the direction columns of d
      for (int z : cyc) {
        CKS(launch_precond_apply<float>(ctx, gr[z], w.Tt + (size_t)goff[z] * nap,
                                        w.Z + (size_t)goff[z] * nap, nap, nap, pm));
        KScope ks_(ctx, KC_KRYLOV);
        k_scatter_add<<<dim3(bg_blocks(nap, 256), gr[z]), 256, 0, st>>>(
            w.Z + (size_t)goff[z] * nap, d, w.map + goff[z], nap);
      }
      for (int z : cyc)
        if (cdone[z]) gdone[z] = 1;
      bool rest = false;
      for (int z : cyc) rest = rest || !gdone[z];
      if (!rest || used >= maxit) break;
      // restart: R_c <- R_c - A M^{-1} (V Y) for the groups still running
      for (int z : cyc) {
        if (gdone[z]) continue;
        CKS(launch_apply<float>(ctx, gr[z], w.Z + (size_t)goff[z] * nap,
                                w.Wb + (size_t)goff[z] * nap, w.apw, nap, pm));
        KScope ks_(ctx, KC_KRYLOV);
        k_sub_cols<<<dim3(bg_blocks(nap, 256), gr[z]), 256, 0, st>>>(
            w.Wb + (size_t)goff[z] * nap, w.Rc + (size_t)goff[z] * nap, nap);
      }
    }
  }
  CK(cudaGetLastError());
  {
    int terr = 0;
    CK(cudaMemcpyFromSymbolAsync(&terr, g_tc_err, sizeof(int), 0, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (terr) {
      ctx->err = "block Krylov update: a tensor-core completion wait ran out";
      return CAVITY_ETIMEOUT;
    }
  }
  return CAVITY_OK;
}
