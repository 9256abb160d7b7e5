// Device building blocks of the shifted-COCG team solver.
//
// Layout used by every kernel: a panel of W right-hand sides is stored as an
// N4 x W array (N4 = 4 * block rows, row-major, complex interleaved), element
// (i, c) at index i * W + c.  A CTA ("team") owns a whole panel; thread t
// always works on column c = t % W (W divides 32 and the block size), so
// per-column partial sums stay in one lane position and reduce without
// atomics, in a fixed order (deterministic results).
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "ffmath.cuh"

namespace gbk {

// Threads per team (CTA).  Several teams share an SM, so that one team's
// barrier and memory stalls are covered by another team's work.
#ifndef GB_TPB
#define GB_TPB 512
#endif
#ifndef GB_UNROLL
#define GB_UNROLL 2
#endif
constexpr int TPB = GB_TPB;
constexpr int kUnroll = GB_UNROLL;  // blocks of a block row in flight per thread
constexpr int NWARP = TPB / 32;
// Two 512-thread teams per SM (64 registers per thread): measured ~20% faster
// than one team with 128 registers on the 1900-orbital chain, despite a few
// spilled registers, because one team's barriers overlap the other's work.
#ifndef GB_MIN_TEAMS
#define GB_MIN_TEAMS ((1024 / GB_TPB) > 0 ? (1024 / GB_TPB) : 1)
#endif
constexpr int MIN_TEAMS_PER_SM = GB_MIN_TEAMS;
// The real recurrence's mixed teams run 512 threads, two per SM, or 1024 (the same
// 64 registers a thread) where a launch has no more panels than SMs: its products
// are bound by load latency with 16 warps on an SM (46 % of issue slots) and by
// issue with 32.  Everything else runs TPB threads.
constexpr int TPB_WIDE = 2 * TPB;
__device__ __forceinline__ int tpb() { return (int)blockDim.x; }
__device__ __forceinline__ int nwarp() { return (int)blockDim.x >> 5; }
constexpr int WMAX = 32;
constexpr int NVMAX = 4;

struct DevMat {
  int n, nb;
  const int* blk_ptr;
  const int* blk_col;
  const double* hb;  // FP64 4x4 blocks, row-major inside a block
  const double* sb;
  const float* hb_hi;  // float-float split of the same blocks: v = hi + lo
  const float* hb_lo;
  const float* sb_hi;
  const float* sb_lo;
  const double* minv;  // inverses of S's diagonal blocks (block Jacobi)
  const float* minv32;
  const int* row_ptr;  // scalar CSR pattern (for R_j and the reductions)
  const int* col_idx;
  const double* h_val;
  const double* s_val;
  const float* h_diag;  // H_ii
  double s_lam_min, s_lam_max;  // spectrum bounds of the block-Jacobi-preconditioned S
  // Block-bidiagonal Cholesky factor of S on 64-row blocks (bf_bw = 0: none).
  // FP64: four [bf_nblk][64][64] arrays, k-major (entry (r, k) at k * 64 + r):
  // D_i^-1, D_i^-T, E_i = D_i^-1 C_i, F_i = D_i^-T C_{i+1}^T.  Mixed path: FP16
  // head / tail fragments of the same tiles (gb::FactorTiles, factor_passes.cuh).
  int bf_bw, bf_nblk;
  const double* bf64;
  const double* bft;  // the FP64 triangles, by row pairs (bc_tri_f64)
  const float* bfm;  // the seed recurrence's TF32 tiles (seed_passes.cuh)
  const uint4* fx;
  int fx_ne, fx_lg;
  float fx_kd[2], fx_ke[2];
  // S^-1 as FP16 fragments (dense_inverse.cuh), di_nt x di_nt tiles of 16 x 16 that
  // 2^di_ex scales back; null: not formed
  const uint4* di;
  int di_nt, di_ex;
};
constexpr int kMmaTileFloatsDev = 52 * 128;  // a TF32 tile: 20 triangular and up to 32 band fragments

// ------------------------------------------------------------ complex FP64
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
__device__ __forceinline__ double2 cinv(double2 b) {
  const double d = b.x * b.x + b.y * b.y;
  return make_double2(b.x / d, -b.y / d);
}
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) { return cmul(a, cinv(b)); }
__device__ __forceinline__ double cabs2(double2 a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ bool cfinite(double2 a) { return isfinite(a.x) && isfinite(a.y); }

// ------------------------------------------------------------ block reduce
struct RedSmem {
  double scal[NVMAX * WMAX];
};

// Sum NV per-thread partials over all threads sharing column c = tid % W.
// Result for (value i, column c) lands in rs.scal[i * WMAX + c].  Fixed order.
// The per-warp partials (warps * NVMAX * 32 doubles) live at the start of the
// kernel's dynamic shared memory, which every team kernel sizes for them.
template <int NV>
__device__ __forceinline__ void block_reduce(double (&v)[NV], int W, RedSmem& rs) {
  extern __shared__ __align__(16) double br_dyn[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int off = W; off < 32; off <<= 1) {
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], off);
  }
  if (lane < W) {
#pragma unroll
    for (int i = 0; i < NV; ++i) br_dyn[(warp * NV + i) * 32 + lane] = v[i];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < NV * W; t += tpb()) {
    const int i = t / W, c = t - i * W;
    double s = 0.0;
    for (int w = 0; w < nwarp(); ++w) s += br_dyn[(w * NV + i) * 32 + c];
    rs.scal[i * WMAX + c] = s;
  }
  __syncthreads();
}

// The same sums for the real recurrence: the warps' partials meet in a shuffle tree
// (one lane per warp) instead of a chain of 16 or 32 dependent FP64 adds, which
// took 2000 of the 26,000 cycles of an update pass.  warps: a power of two.
template <int NV>
__device__ __forceinline__ void block_reduce_tree(double (&v)[NV], int W, RedSmem& rs) {
  extern __shared__ __align__(16) double br_dyn[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = nwarp();
  for (int off = W; off < 32; off <<= 1) {
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], off);
  }
  if (lane < W) {
#pragma unroll
    for (int i = 0; i < NV; ++i) br_dyn[(i * W + lane) * nw + warp] = v[i];
  }
  __syncthreads();
  // whole warps: NV * W * nw is a multiple of 32 for every W >= 1 (nw >= 16, NV = 2)
  static_assert(NV % 2 == 0, "whole warps take the partials");
  for (int t = threadIdx.x; t < NV * W * nw; t += tpb()) {
    double s = br_dyn[t];
    for (int off = nw >> 1; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    const int o = t / nw;
    if (t - o * nw == 0) rs.scal[(o / W) * WMAX + o % W] = s;
  }
  __syncthreads();
}

// The same for two compensated accumulators per thread (the mixed path's dots): the
// lanes of a warp meet in FP32 pairs and FP64 starts with one lane per warp and
// column.  A warp's FP64 instruction holds its scheduler for 64 cycles on GB300, so
// converting and adding in every lane cost 6000 cycles a reduction.
__device__ __forceinline__ void acc_xor_combine(gbff::acc& a, int off) {
  const float oh = __shfl_xor_sync(0xffffffffu, a.hi, off);
  const float oe = __shfl_xor_sync(0xffffffffu, a.err, off);
  const gbff::ff sm = gbff::two_sum(a.hi, oh);
  a.hi = sm.hi;
  a.err = __fadd_rn(__fadd_rn(a.err, oe), sm.lo);
}
__device__ __forceinline__ void block_reduce_acc(gbff::acc d0, gbff::acc d1, int W, RedSmem& rs) {
  extern __shared__ __align__(16) double br_dyn[];
  float2* part = reinterpret_cast<float2*>(br_dyn);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = nwarp();
  for (int off = W; off < 32; off <<= 1) {
    acc_xor_combine(d0, off);
    acc_xor_combine(d1, off);
  }
  if (lane < W) {
    part[lane * nw + warp] = make_float2(d0.hi, d0.err);
    part[(W + lane) * nw + warp] = make_float2(d1.hi, d1.err);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 2 * W * nw; t += tpb()) {  // whole warps
    const float2 p = part[t];
    double s = (double)p.x + (double)p.y;
    for (int off = nw >> 1; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    const int o = t / nw;
    if (t - o * nw == 0) rs.scal[(o / W) * WMAX + o % W] = s;
  }
  __syncthreads();
}

// ------------------------------------------------------------ BSR block-row products
// acc[r] = sum over stored blocks (I, J) of A_IJ[r][t] * x[4J + t][c]; FP64.
__device__ __forceinline__ void bsr_row_d(const DevMat& m, const double* __restrict__ A,
                                          const double2* __restrict__ x, int W, int c, int I,
                                          double2 (&acc)[4]) {
#pragma unroll
  for (int r = 0; r < 4; ++r) acc[r] = make_double2(0.0, 0.0);
  const int b1 = m.blk_ptr[I + 1];
#pragma unroll kUnroll
  for (int b = m.blk_ptr[I]; b < b1; ++b) {
    const int J = m.blk_col[b];
    const double2* xr = x + (size_t)(4 * J) * W + c;
    double2 xv[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) xv[t] = xr[(size_t)t * W];
    const double2* ab = reinterpret_cast<const double2*>(A + (size_t)b * 16);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const double2 a01 = __ldg(ab + 2 * r), a23 = __ldg(ab + 2 * r + 1);
      acc[r].x = fma(a01.x, xv[0].x, acc[r].x);
      acc[r].y = fma(a01.x, xv[0].y, acc[r].y);
      acc[r].x = fma(a01.y, xv[1].x, acc[r].x);
      acc[r].y = fma(a01.y, xv[1].y, acc[r].y);
      acc[r].x = fma(a23.x, xv[2].x, acc[r].x);
      acc[r].y = fma(a23.x, xv[2].y, acc[r].y);
      acc[r].x = fma(a23.y, xv[3].x, acc[r].x);
      acc[r].y = fma(a23.y, xv[3].y, acc[r].y);
    }
  }
}

// FP32 matrix (hi part) times FP32 complex vector, FP32 accumulation.
__device__ __forceinline__ void bsr_row_f(const DevMat& m, const float* __restrict__ A,
                                          const float2* __restrict__ x, int W, int c, int I,
                                          float2 (&acc)[4]) {
#pragma unroll
  for (int r = 0; r < 4; ++r) acc[r] = make_float2(0.f, 0.f);
  const int b1 = m.blk_ptr[I + 1];
#pragma unroll kUnroll
  for (int b = m.blk_ptr[I]; b < b1; ++b) {
    const int J = m.blk_col[b];
    const float2* xr = x + (size_t)(4 * J) * W + c;
    float2 xv[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) xv[t] = xr[(size_t)t * W];
    const float4* ab = reinterpret_cast<const float4*>(A + (size_t)b * 16);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 a = __ldg(ab + r);
      acc[r].x = fmaf(a.x, xv[0].x, acc[r].x);
      acc[r].y = fmaf(a.x, xv[0].y, acc[r].y);
      acc[r].x = fmaf(a.y, xv[1].x, acc[r].x);
      acc[r].y = fmaf(a.y, xv[1].y, acc[r].y);
      acc[r].x = fmaf(a.z, xv[2].x, acc[r].x);
      acc[r].y = fmaf(a.z, xv[2].y, acc[r].y);
      acc[r].x = fmaf(a.w, xv[3].x, acc[r].x);
      acc[r].y = fmaf(a.w, xv[3].y, acc[r].y);
    }
  }
}

// FP32 matrix (hi part) times the hi parts of a float-float complex vector
// (float4 {re.hi, re.lo, im.hi, im.lo}), FP32 accumulation: the unrefined
// FP32 product (flags bit 5 of the mixed path).
__device__ __forceinline__ void bsr_row_fhi(const DevMat& m, const float* __restrict__ A,
                                            const float4* __restrict__ x, int W, int c, int I, float2 (&acc)[4]) {
#pragma unroll
  for (int r = 0; r < 4; ++r) acc[r] = make_float2(0.f, 0.f);
  const int b1 = m.blk_ptr[I + 1];
#pragma unroll kUnroll
  for (int b = m.blk_ptr[I]; b < b1; ++b) {
    const int J = m.blk_col[b];
    const float4* xr = x + (size_t)(4 * J) * W + c;
    float2 xv[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const float4 v = xr[(size_t)t * W];
      xv[t] = make_float2(v.x, v.z);
    }
    const float4* ab = reinterpret_cast<const float4*>(A + (size_t)b * 16);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 a = __ldg(ab + r);
      acc[r].x = fmaf(a.x, xv[0].x, fmaf(a.y, xv[1].x, fmaf(a.z, xv[2].x, fmaf(a.w, xv[3].x, acc[r].x))));
      acc[r].y = fmaf(a.x, xv[0].y, fmaf(a.y, xv[1].y, fmaf(a.z, xv[2].y, fmaf(a.w, xv[3].y, acc[r].y))));
    }
  }
}

// float-float matrix (hi + lo) times float-float complex vector, compensated
// accumulation: acc_re[r] / acc_im[r] hold the row sums as hi + err.
__device__ __forceinline__ void bsr_row_ff(const DevMat& m, const float* __restrict__ Ahi,
                                           const float* __restrict__ Alo, const float4* __restrict__ x,
                                           int W, int c, int I, gbff::acc (&are)[4], gbff::acc (&aim)[4]) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    gbff::acc_init(are[r]);
    gbff::acc_init(aim[r]);
  }
  const int b1 = m.blk_ptr[I + 1];
#pragma unroll kUnroll
  for (int b = m.blk_ptr[I]; b < b1; ++b) {
    const int J = m.blk_col[b];
    const float4* xr = x + (size_t)(4 * J) * W + c;
    float4 xv[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) xv[t] = xr[(size_t)t * W];
    const float4* ah = reinterpret_cast<const float4*>(Ahi + (size_t)b * 16);
    const float4* al = reinterpret_cast<const float4*>(Alo + (size_t)b * 16);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 h = __ldg(ah + r), l = __ldg(al + r);
      const float hv[4] = {h.x, h.y, h.z, h.w};
      const float lv[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const gbff::ff a = {hv[t], lv[t]};
        gbff::acc_mul_add(are[r], a, gbff::ff{xv[t].x, xv[t].y});
        gbff::acc_mul_add(aim[r], a, gbff::ff{xv[t].z, xv[t].w});
      }
    }
  }
}

// float-float matrix times FP32 complex vector (x exact in float), compensated.
__device__ __forceinline__ void bsr_row_ffx(const DevMat& m, const float* __restrict__ Ahi,
                                            const float* __restrict__ Alo, const float2* __restrict__ x,
                                            int W, int c, int I, gbff::acc (&are)[4], gbff::acc (&aim)[4]) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    gbff::acc_init(are[r]);
    gbff::acc_init(aim[r]);
  }
  const int b1 = m.blk_ptr[I + 1];
#pragma unroll kUnroll
  for (int b = m.blk_ptr[I]; b < b1; ++b) {
    const int J = m.blk_col[b];
    const float2* xr = x + (size_t)(4 * J) * W + c;
    float2 xv[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) xv[t] = xr[(size_t)t * W];
    const float4* ah = reinterpret_cast<const float4*>(Ahi + (size_t)b * 16);
    const float4* al = reinterpret_cast<const float4*>(Alo + (size_t)b * 16);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 h = __ldg(ah + r), l = __ldg(al + r);
      const float hv[4] = {h.x, h.y, h.z, h.w};
      const float lv[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const gbff::ff a = {hv[t], lv[t]};
        gbff::acc_mul_add(are[r], a, xv[t].x);
        gbff::acc_mul_add(aim[r], a, xv[t].y);
      }
    }
  }
}


// ------------------------------------------------------------ one scalar row per thread
// The real recurrence's products: thread = (row i = 4 I + r, column pair c), that
// is element e = i W + c of the panel, so results and dots are coalesced.  The four
// rows of a block share its x loads through the warp (same addresses), and each
// loads its own matrix row.  Against one block row per thread (above) a panel has
// four times the threads at work and a quarter of the accumulators each: the team
// waits on load latency (ncu: 29 % of issue slots used with one team per SM), and
// two blocks in flight fit the 64 registers without spills.  Together with the wide
// teams and the cheaper reductions: an iteration of 912 orbitals, all columns, 375 ->
// 242 us, of 24 columns of 1900 419 -> 257 us.
// float-float row times a float-float vector (float4 pairs).
__device__ __forceinline__ void row_ff(const DevMat& m, const float* __restrict__ Ahi, const float* __restrict__ Alo,
                                       const float4* x, int W, int c, int row, gbff::acc& a0, gbff::acc& a1) {
  gbff::acc_init(a0);
  gbff::acc_init(a1);
  const float4* ah = reinterpret_cast<const float4*>(Ahi) + (row & 3);
  const float4* al = reinterpret_cast<const float4*>(Alo) + (row & 3);
  const int I = row >> 2, b1 = m.blk_ptr[I + 1];
#pragma unroll 2
  for (int b = m.blk_ptr[I]; b < b1; ++b) {
    const float4* xr = x + (size_t)(4 * m.blk_col[b]) * W + c;
    const float4 h = __ldg(ah + 4 * (size_t)b), l = __ldg(al + 4 * (size_t)b);
    float4 xv[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) xv[t] = xr[t * W];
    const float hv[4] = {h.x, h.y, h.z, h.w}, lv[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      gbff::acc_mul_add(a0, gbff::ff{hv[t], lv[t]}, gbff::ff{xv[t].x, xv[t].y});
      gbff::acc_mul_add(a1, gbff::ff{hv[t], lv[t]}, gbff::ff{xv[t].z, xv[t].w});
    }
  }
}

// float-float row times an FP32 vector (float2 pairs), compensated.
__device__ __forceinline__ void row_ffx(const DevMat& m, const float* __restrict__ Ahi, const float* __restrict__ Alo,
                                        const float2* x, int W, int c, int row, gbff::acc& a0, gbff::acc& a1) {
  gbff::acc_init(a0);
  gbff::acc_init(a1);
  const float4* ah = reinterpret_cast<const float4*>(Ahi) + (row & 3);
  const float4* al = reinterpret_cast<const float4*>(Alo) + (row & 3);
  const int I = row >> 2, b1 = m.blk_ptr[I + 1];
#pragma unroll 2
  for (int b = m.blk_ptr[I]; b < b1; ++b) {
    const float2* xr = x + (size_t)(4 * m.blk_col[b]) * W + c;
    const float4 h = __ldg(ah + 4 * (size_t)b), l = __ldg(al + 4 * (size_t)b);
    float2 xv[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) xv[t] = xr[t * W];
    const float hv[4] = {h.x, h.y, h.z, h.w}, lv[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      gbff::acc_mul_add(a0, gbff::ff{hv[t], lv[t]}, xv[t].x);
      gbff::acc_mul_add(a1, gbff::ff{hv[t], lv[t]}, xv[t].y);
    }
  }
}

// FP32 row (the heads) times an FP32 vector: float2 pairs, or the heads of float4 pairs.
template <typename XV>
__device__ __forceinline__ float2 row_f(const DevMat& m, const float* __restrict__ A, const XV* x, int W, int c,
                                        int row) {
  float2 acc = make_float2(0.f, 0.f);
  const float4* ah = reinterpret_cast<const float4*>(A) + (row & 3);
  const int I = row >> 2, b1 = m.blk_ptr[I + 1];
#pragma unroll 4
  for (int b = m.blk_ptr[I]; b < b1; ++b) {
    const XV* xr = x + (size_t)(4 * m.blk_col[b]) * W + c;
    const float4 h = __ldg(ah + 4 * (size_t)b);
    const float hv[4] = {h.x, h.y, h.z, h.w};
    XV xv[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) xv[t] = xr[t * W];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if constexpr (sizeof(XV) == 16) {
        acc.x = fmaf(hv[t], xv[t].x, acc.x);
        acc.y = fmaf(hv[t], xv[t].z, acc.y);
      } else {
        acc.x = fmaf(hv[t], xv[t].x, acc.x);
        acc.y = fmaf(hv[t], xv[t].y, acc.y);
      }
    }
  }
  return acc;
}

__device__ __forceinline__ double2 row_d(const DevMat& m, const double* __restrict__ A, const double2* x, int W, int c,
                                         int row) {
  double2 acc = make_double2(0.0, 0.0);
  const double2* ar = reinterpret_cast<const double2*>(A) + 2 * (row & 3);
  const int I = row >> 2, b1 = m.blk_ptr[I + 1];
#pragma unroll 2
  for (int b = m.blk_ptr[I]; b < b1; ++b) {
    const double2* xr = x + (size_t)(4 * m.blk_col[b]) * W + c;
    const double2 a01 = __ldg(ar + 8 * (size_t)b), a23 = __ldg(ar + 8 * (size_t)b + 1);
    const double2 x0 = xr[0], x1 = xr[W], x2 = xr[2 * W], x3 = xr[3 * W];
    acc.x = fma(a01.x, x0.x, acc.x);
    acc.y = fma(a01.x, x0.y, acc.y);
    acc.x = fma(a01.y, x1.x, acc.x);
    acc.y = fma(a01.y, x1.y, acc.y);
    acc.x = fma(a23.x, x2.x, acc.x);
    acc.y = fma(a23.x, x2.y, acc.y);
    acc.x = fma(a23.y, x3.x, acc.x);
    acc.y = fma(a23.y, x3.y, acc.y);
  }
  return acc;
}

}  // namespace gbk
