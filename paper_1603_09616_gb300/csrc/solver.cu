// C ABI of the GB300 shifted Green's-function library (declared in gbgreen.h).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <functional>
#include <memory>
#include <vector>

#include "gb_internal.h"
#include "team_kernels.cuh"
#include "wavepacket_cluster.cuh"

namespace gb {

static thread_local char g_err[512];

gb_status fail(gb_status st, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof g_err, fmt, ap);
  va_end(ap);
  return st;
}
void clear_error() { g_err[0] = 0; }

static gb_status cuda_fail(cudaError_t e, const char* what) {
  return fail(GB_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define GB_CUDA(call)                                 \
  do {                                                \
    cudaError_t e_ = (call);                          \
    if (e_ != cudaSuccess) return cuda_fail(e_, #call); \
  } while (0)

static size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// Caller-owned device buffers are read and written with vector accesses of
// their element size (complex doubles as 16-byte double2): a pointer off that
// boundary is an error, found here instead of as a misaligned access.
static bool misaligned(const void* p, size_t bytes) { return p && (reinterpret_cast<uintptr_t>(p) % bytes) != 0; }
static gb_status check_outputs(const gb_outputs* o) {
  if (misaligned(o->ldos, 8) || misaligned(o->rho, 8) || misaligned(o->edm, 8) || misaligned(o->q, 8) ||
      misaligned(o->e_loc, 8) || misaligned(o->resid, 8) || misaligned(o->iters, 4) ||
      misaligned(o->inner_iters, 4) || misaligned(o->col_status, 4) || misaligned(o->g_proj, 16))
    return fail(GB_EINVAL, "an output is not aligned to its element (g_proj: 16 bytes)");
  return GB_OK;
}

}  // namespace gb

struct gb_matrix {
  int device = 0;
  int64_t n = 0, nb = 0, nnz = 0, nnzb = 0;
  int32_t max_row = 0;
  std::vector<int64_t> h_row_ptr;  // host copy of the pattern's row pointers
  void* base = nullptr;
  gbk::DevMat dm{};
};

namespace gb {
const gbk::DevMat* devmat_of(const gb_matrix* m) { return &m->dm; }
}  // namespace gb

using namespace gb;

// ------------------------------------------------------------ standalone SpMM
namespace {

// Narrow FP32 panels (W = 1, 2, 4): one warp per block row, lane l owns row
// r = l % 4 of the stored blocks b0 + l / 4, b0 + l / 4 + 8, ...  The lanes of
// a warp read 8 whole consecutive blocks per step (512 contiguous bytes: each
// 32-byte sector requested once), the 4 lanes of a block share its x gather
// (same addresses, one request), and every lane accumulates a single row, so
// the reduction is three xor-shuffle levels over the 8 block slots.  Requires
// x 16-byte aligned (float4 loads of the 4 x W gathered entries).
// acc[c] += (row of a block) . x[4 rows, column c]; the complex x entry
// (row t, column c) is float2 number t * WC + c of the gathered float4s.
template <int WC>
__device__ __forceinline__ void quad_fma(const float4& a, const float4 (&xv)[2 * WC], float2 (&acc)[WC]) {
#pragma unroll
  for (int c = 0; c < WC; ++c) {
    float xr[4], xi[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int f = t * WC + c;
      const float4 q = xv[f >> 1];
      xr[t] = (f & 1) ? q.z : q.x;
      xi[t] = (f & 1) ? q.w : q.y;
    }
    acc[c].x = fmaf(a.x, xr[0], fmaf(a.y, xr[1], fmaf(a.z, xr[2], fmaf(a.w, xr[3], acc[c].x))));
    acc[c].y = fmaf(a.x, xi[0], fmaf(a.y, xi[1], fmaf(a.z, xi[2], fmaf(a.w, xi[3], acc[c].y))));
  }
}

// The kernel is bound by loads in flight: the block columns are fetched a
// step ahead, W = 1 keeps two 8-block steps in flight per lane and W = 2 one,
// at 40 registers (48 warps per SM) without spills.
// RAG (n not a multiple of 4): x ends inside the last block column's four rows, whose
// missing ones are zero; read with guards there instead of from a padded copy of x
// (an allocation, two copies and a free: 14 of 23 us at 23,750 rows, and 200 us where
// the call was waited for, because the pool gave its memory back).
// X8: x on an 8-byte boundary only (read entry by entry).
template <int WC, bool RAG, bool X8 = false>
__global__ void __launch_bounds__(256, 6)
    spmm_quad_kernel(const gbk::DevMat m, const float* __restrict__ A, const float2* __restrict__ x,
                     float2* __restrict__ y) {
  const long long I = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  if (I >= m.nb) return;  // uniform per warp
  const int lane = threadIdx.x & 31, r = lane & 3, s = lane >> 2;
  constexpr int U = WC == 1 ? 2 : 1;  // steps of 8 blocks in flight per lane
  constexpr int NQ = 2 * WC;  // float4 per gathered 4 x WC complex x block
  float2 acc[WC];
#pragma unroll
  for (int c = 0; c < WC; ++c) acc[c] = make_float2(0.f, 0.f);
  const int b1 = m.blk_ptr[I + 1];
  const float4* __restrict__ A4 = reinterpret_cast<const float4*>(A);
  const float4* __restrict__ X4 = reinterpret_cast<const float4*>(x);
  auto guarded = [&](int J, float4 (&xv)[NQ]) {  // float4 q: complex entries 2 q and 2 q + 1 of the 4 x WC
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int r0 = 4 * J + 2 * q / WC, r1 = 4 * J + (2 * q + 1) / WC;
      const float2 z = make_float2(0.f, 0.f);
      const float2 u = !RAG || r0 < m.n ? x[(size_t)4 * J * WC + 2 * q] : z;
      const float2 v = !RAG || r1 < m.n ? x[(size_t)4 * J * WC + 2 * q + 1] : z;
      xv[q] = make_float4(u.x, u.y, v.x, v.y);
    }
  };
  int b = m.blk_ptr[I] + s;
  // block columns one step ahead: the x gathers of a step then wait for one
  // memory round trip, not two (column index, then x)
  int Jn[U];
#pragma unroll
  for (int u = 0; u < U; ++u) Jn[u] = b + 8 * u < b1 ? __ldcs(m.blk_col + b + 8 * u) : 0;
  for (; b + 8 * (U - 1) < b1; b += 8 * U) {
    int J[U];
    float4 a[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      J[u] = Jn[u];
      const int bn = b + 8 * U + 8 * u;
      Jn[u] = bn < b1 ? __ldcs(m.blk_col + bn) : 0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) a[u] = __ldcs(A4 + (size_t)(b + 8 * u) * 4 + r);
    float4 xv[U][NQ];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if constexpr (X8) {
        guarded(J[u], xv[u]);
      } else {
        if (RAG && J[u] == m.nb - 1) {
          guarded(J[u], xv[u]);
          continue;
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) xv[u][q] = __ldg(X4 + (size_t)J[u] * NQ + q);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) quad_fma<WC>(a[u], xv[u], acc);
  }
  for (; b < b1; b += 8) {
    const int J = Jn[0];  // the loop above leaves the next step's columns in Jn
    const float4 a = __ldcs(A4 + (size_t)b * 4 + r);
#pragma unroll
    for (int u = 0; u + 1 < U; ++u) Jn[u] = Jn[u + 1];
    float4 xv[NQ];
    if (X8 || (RAG && J == m.nb - 1)) {
      guarded(J, xv);
    } else {
#pragma unroll
      for (int q = 0; q < NQ; ++q) xv[q] = __ldg(X4 + (size_t)J * NQ + q);
    }
    quad_fma<WC>(a, xv, acc);
  }
#pragma unroll
  for (int off = 4; off < 32; off <<= 1)
#pragma unroll
    for (int c = 0; c < WC; ++c) {
      acc[c].x += __shfl_xor_sync(0xffffffffu, acc[c].x, off);
      acc[c].y += __shfl_xor_sync(0xffffffffu, acc[c].y, off);
    }
  if (s == 0 && 4 * I + r < m.n) {
#pragma unroll
    for (int c = 0; c < WC; ++c) y[(size_t)(4 * I + r) * WC + c] = acc[c];
  }
}

// FP64, any width: threads own (row, column) outputs, consecutive threads consecutive
// columns of a row, and walk the row's pattern entries (scalar CSR); W = 1 and 2 split
// a row over E = 4 and 2 lanes that meet in shuffles.  The product is bound by the FP64
// pipe (1/64 of the FP32 rate), so what counts is the number of FMAs: the pattern's
// entries, not the 4x4 blocks' (a third of which is padding on the bundles).  The bytes
// are those of the blocks: 12 an entry against 8 / fill.  41,040-orbital bundle, W = 8:
// blocks 240 us, entries 167 us (W = 1: 43 and 31).
template <int E>
__global__ void __launch_bounds__(256)
    spmm_csr_d_kernel(const gbk::DevMat m, const double* __restrict__ A, int W, const double2* __restrict__ x,
                      double2* __restrict__ y) {
  const long long o = (blockIdx.x * 256LL + threadIdx.x) / E;  // output row * W + column
  const int slot = threadIdx.x % E;
  const bool in = o < (long long)m.n * W;
  const int row = in ? (int)(o / W) : 0, c = in ? (int)(o - (long long)row * W) : 0;
  const int e1 = in ? m.row_ptr[row + 1] : 0;
  double2 acc = make_double2(0.0, 0.0);
#pragma unroll 4
  for (int e = (in ? m.row_ptr[row] : 0) + slot; e < e1; e += E) {
    const double a = __ldg(A + e);
    const double2 v = __ldg(x + (size_t)__ldg(m.col_idx + e) * W + c);
    acc.x = fma(a, v.x, acc.x);
    acc.y = fma(a, v.y, acc.y);
  }
#pragma unroll
  for (int k = E / 2; k > 0; k >>= 1) {
    acc.x += __shfl_xor_sync(0xffffffffu, acc.x, k);
    acc.y += __shfl_xor_sync(0xffffffffu, acc.y, k);
  }
  if (in && slot == 0) y[o] = acc;
}

// Wide FP32 panels (W = 4..64 in powers of two): one warp
// per block row, split into G = 32 / CL groups of CL lanes; group g takes the
// blocks b0 + g + G k, and lane c of a group owns columns [c * PC, (c+1) * PC)
// of the panel (PC = 2 complex columns per lane, read and written as one float4).  A block's values are read by every lane of its
// group at one address (a broadcast), its x rows by the group as contiguous
// runs, and each value feeds PC complex columns from registers.  The groups
// then add up through xor shuffles.  Requires x and y 16-byte aligned.
// The kernel waits on loads (ncu at W = 8: long-scoreboard stalls dominate),
// so it keeps one step in flight per lane at <= 64 registers, which lets 32
// warps share an SM (two steps at 106 registers left 11 warps active).
template <int CL, bool RAG>
__global__ void __launch_bounds__(256, 4)
    spmm_wide_kernel(const gbk::DevMat m, const float* __restrict__ A, const float4* __restrict__ x,
                     float4* __restrict__ y) {
  constexpr int G = 32 / CL;
  const long long I = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  if (I >= m.nb) return;
  const int lane = threadIdx.x & 31, g = lane / CL, c = lane - g * CL;
  float4 acc[4];  // row r: (re, im) of columns 2c and 2c + 1
#pragma unroll
  for (int r = 0; r < 4; ++r) acc[r] = make_float4(0.f, 0.f, 0.f, 0.f);
  const float4* __restrict__ A4 = reinterpret_cast<const float4*>(A);
  auto step = [&](const float4 (&a)[4], const float4 (&xv)[4]) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float ar[4] = {a[r].x, a[r].y, a[r].z, a[r].w};
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        acc[r].x = fmaf(ar[t], xv[t].x, acc[r].x);
        acc[r].y = fmaf(ar[t], xv[t].y, acc[r].y);
        acc[r].z = fmaf(ar[t], xv[t].z, acc[r].z);
        acc[r].w = fmaf(ar[t], xv[t].w, acc[r].w);
      }
    }
  };
  auto fetch = [&](int row) {
    return !RAG || row < m.n ? __ldg(x + (size_t)row * CL + c) : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  const int b1 = m.blk_ptr[I + 1];
  int b = m.blk_ptr[I] + g;
  constexpr int U = 1;
  int Jn[U];  // block columns one step ahead (one round trip per step)
#pragma unroll
  for (int u = 0; u < U; ++u) Jn[u] = b + G * u < b1 ? __ldcs(m.blk_col + b + G * u) : 0;
  for (; b + G * (U - 1) < b1; b += G * U) {
    int J[U];
    float4 a[U][4], xv[U][4];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      J[u] = Jn[u];
      const int bn = b + G * U + G * u;
      Jn[u] = bn < b1 ? __ldcs(m.blk_col + bn) : 0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int r = 0; r < 4; ++r) a[u][r] = __ldcs(A4 + (size_t)(b + G * u) * 4 + r);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int t = 0; t < 4; ++t) xv[u][t] = fetch(4 * J[u] + t);
#pragma unroll
    for (int u = 0; u < U; ++u) step(a[u], xv[u]);
  }
  for (; b < b1; b += G) {
    const int J = Jn[0];
#pragma unroll
    for (int u = 0; u + 1 < U; ++u) Jn[u] = Jn[u + 1];
    float4 a[4], xv[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) a[r] = __ldcs(A4 + (size_t)b * 4 + r);
#pragma unroll
    for (int t = 0; t < 4; ++t) xv[t] = fetch(4 * J + t);
    step(a, xv);
  }
#pragma unroll
  for (int off = CL; off < 32; off <<= 1)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      acc[r].x += __shfl_xor_sync(0xffffffffu, acc[r].x, off);
      acc[r].y += __shfl_xor_sync(0xffffffffu, acc[r].y, off);
      acc[r].z += __shfl_xor_sync(0xffffffffu, acc[r].z, off);
      acc[r].w += __shfl_xor_sync(0xffffffffu, acc[r].w, off);
    }
  if (g == 0) {
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (4 * I + r < m.n) y[(size_t)(4 * I + r) * CL + c] = acc[r];
  }
}

// FP32, what the kernels above do not take (other widths, x or y off a 16-byte
// boundary).  W <= 8: one warp per block row, its lanes split as columns x block slots
// (four blocks in flight a lane); wider: one thread per (block row, column).  One thread
// per (row, column) took 1.5 to 3.6 times as long at W = 3 .. 33 (41,040 orbitals).
template <bool RAG>
__global__ void __launch_bounds__(256)
    spmm_any_kernel(const gbk::DevMat m, const float* __restrict__ A, int W, const float2* __restrict__ x,
                    float2* __restrict__ y) {
  float2 acc[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) acc[r] = make_float2(0.f, 0.f);
  const float4* __restrict__ A4 = reinterpret_cast<const float4*>(A);
  auto fetch = [&](int row, int c) {
    return !RAG || row < m.n ? x[(size_t)row * W + c] : make_float2(0.f, 0.f);
  };
  auto mul = [&](const float4 (&a)[4], const float2 (&v)[4]) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      acc[r].x = fmaf(a[r].x, v[0].x, fmaf(a[r].y, v[1].x, fmaf(a[r].z, v[2].x, fmaf(a[r].w, v[3].x, acc[r].x))));
      acc[r].y = fmaf(a[r].x, v[0].y, fmaf(a[r].y, v[1].y, fmaf(a[r].z, v[2].y, fmaf(a[r].w, v[3].y, acc[r].y))));
    }
  };
  const long long at = blockIdx.x * 256LL + threadIdx.x;
  int I, c, b, S = 1;
  bool store = true;
  if (W <= 8) {
    const int Wp = W <= 1 ? 1 : (W <= 2 ? 2 : (W <= 4 ? 4 : 8)), lane = (int)(at & 31);
    I = (int)(at >> 5);
    if (I >= m.nb) return;  // uniform per warp
    c = lane % Wp;
    S = 32 / Wp;
    b = m.blk_ptr[I] + lane / Wp;
    store = lane < W;
    if (c >= W) b = m.blk_ptr[I + 1];  // no column: only the shuffles
  } else {
    if (at >= (long long)m.nb * W) return;
    I = (int)(at / W);
    c = (int)(at - (long long)I * W);
    b = m.blk_ptr[I];
  }
  const int b1 = m.blk_ptr[I + 1];
  for (; b + 3 * S < b1; b += 4 * S) {
    int J[4];
    float4 a[4][4];
    float2 v[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u) J[u] = __ldg(m.blk_col + b + u * S);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
#pragma unroll
      for (int r = 0; r < 4; ++r) a[u][r] = __ldg(A4 + (size_t)(b + u * S) * 4 + r);
#pragma unroll
      for (int t = 0; t < 4; ++t) v[u][t] = fetch(4 * J[u] + t, c);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) mul(a[u], v[u]);
  }
  for (; b < b1; b += S) {
    const int J = __ldg(m.blk_col + b);
    float4 a[4];
    float2 v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) a[r] = __ldg(A4 + (size_t)b * 4 + r);
#pragma unroll
    for (int t = 0; t < 4; ++t) v[t] = fetch(4 * J + t, c);
    mul(a, v);
  }
  if (W <= 8) {
    for (int off = 32 / S; off < 32; off <<= 1) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        acc[r].x += __shfl_xor_sync(0xffffffffu, acc[r].x, off);
        acc[r].y += __shfl_xor_sync(0xffffffffu, acc[r].y, off);
      }
    }
  }
  if (!store) return;
#pragma unroll
  for (int r = 0; r < 4; ++r)
    if (4 * I + r < m.n) y[(size_t)(4 * I + r) * W + c] = acc[r];
}

}  // namespace

// ------------------------------------------------------------ what a matrix keeps beside FP64
namespace {

// Float-float splits v = hi + lo (lo may be null: hi alone) of n FP64 values.
__global__ void split_kernel(const double* __restrict__ v, size_t n, float* __restrict__ hi, float* __restrict__ lo) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const double x = v[i];
    const float h = (float)x;
    hi[i] = h;
    if (lo) lo[i] = (float)(x - (double)h);
  }
}

// The onsite energies (every row of the pattern has its diagonal entry).
__global__ void diag_kernel(const gbk::DevMat m, float* __restrict__ d) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= m.n) return;
  int lo = m.row_ptr[i], hi = m.row_ptr[i + 1];
  while (lo < hi) {  // first column >= i of the sorted row
    const int mid = (lo + hi) >> 1;
    if (m.col_idx[mid] < i) lo = mid + 1;
    else hi = mid;
  }
  d[i] = lo < m.row_ptr[i + 1] && m.col_idx[lo] == i ? (float)m.h_val[lo] : 0.f;
}

// The factor's tiles in MMA fragment order, one block of threads per 64-row block
// and direction.  Element (r, k) of a 64 x 64 factor block lies at k * 64 + r.
//
// FP16 tiles (factor_passes.cuh): fragments of 16 x 16 (mi, kk), the entries scaled
// to below 2^4, 32 lanes x 4 words of FP16 heads and then the same of tails.  Lane
// l = 4 g + t holds in word q row g + 8 (q & 1) and the column pair w = t + 4 (q >> 1),
// a pair being columns w and w + 8: the order in which the passes pack the vector's
// rows.  First the triangle's (FWD: kk <= mi, by mi then kk; BWD: kk >= mi), then the
// band's (E: its last ne column steps; F: its first), by mi.
//
// TF32 tiles (seed_passes.cuh): fragments of 16 x 8 (mi, ks), lane l's word q is
// A(g + 8 (q & 1), t + 4 (q >> 1)); first the triangle's (FWD: mi >= ks / 2, by ks
// then mi; BWD: mi <= ks / 2), then the band's (E: ks from (64 - bw) / 8; F: ks below
// ceil(bw / 8)), by ks.
struct TileArgs {
  const double* bf;
  size_t part;
  int n, bw, ne;
  float sd[2], se[2];
  uint32_t* fx;
  float* tf;
};
__global__ void __launch_bounds__(256) tile_kernel(TileArgs a) {
  const int blk = blockIdx.x >> 1, dir = blockIdx.x & 1;
  const double* D = a.bf + dir * a.part + (size_t)blk * 4096;
  const double* E = a.bf + (2 + dir) * a.part + (size_t)blk * 4096;
  uint32_t* fx = a.fx + (size_t)blockIdx.x * (10 + 4 * a.ne) * 256;
  for (int e = threadIdx.x; a.fx && e < (10 + 4 * a.ne) * 128; e += 256) {
    const int f = e >> 7, l = (e & 127) >> 2, q = e & 3;
    int mi, kk;
    if (f < 10) {
      mi = 0;
      while (f >= (dir ? 4 * (mi + 1) - (mi + 1) * mi / 2 : (mi + 1) * (mi + 2) / 2)) ++mi;
      kk = dir ? f - (4 * mi - mi * (mi - 1) / 2) + mi : f - mi * (mi + 1) / 2;
    } else {
      mi = (f - 10) / a.ne;
      kk = (f - 10) % a.ne + (dir ? 0 : 4 - a.ne);
    }
    const double* M = f < 10 ? D : E;
    const double sc = f < 10 ? a.sd[dir] : a.se[dir];
    const int r = 16 * mi + (l >> 2) + 8 * (q & 1), k = 16 * kk + (l & 3) + 4 * (q >> 1);
    // the padding's unit diagonal would not fit the scale; its rows of the vector are zero
    const bool in = 64 * blk + r < a.n;
    uint32_t h, t;
    gbk::split_f16(in ? (float)(M[k * 64 + r] * sc) : 0.f, in ? (float)(M[(k + 8) * 64 + r] * sc) : 0.f, h, t);
    fx[(size_t)f * 256 + l * 4 + q] = h;
    fx[(size_t)f * 256 + 128 + l * 4 + q] = t;
  }
  float* tf = a.tf + (size_t)blockIdx.x * gbk::kMmaTileFloatsDev;
  const int ks0 = dir ? 0 : (64 - a.bw) / 8, n2 = dir ? (a.bw + 7) / 8 : 8 - ks0;
  for (int e = threadIdx.x; e < (20 + 4 * n2) * 128; e += 256) {
    const int f = e >> 7, l = (e & 127) >> 2, q = e & 3;
    int mi, ks;
    if (f < 20) {
      int left = f;
      for (ks = 0;; ++ks) {
        const int c = dir ? ks / 2 + 1 : 4 - ks / 2;
        if (left < c) break;
        left -= c;
      }
      mi = dir ? left : ks / 2 + left;
    } else {
      ks = ks0 + (f - 20) / 4;
      mi = (f - 20) & 3;
    }
    const int r = 16 * mi + (l >> 2) + 8 * (q & 1), k = 8 * ks + (l & 3) + 4 * (q >> 1);
    tf[e] = (float)(f < 20 ? D : E)[k * 64 + r];
  }
}

// The FP64 solve's triangles by row pairs (bc_tri_f64), one block of threads per 64-row
// block and direction.
__global__ void __launch_bounds__(256) tri_pack_kernel(const double* __restrict__ bf, size_t part,
                                                       double* __restrict__ out) {
  const int blk = blockIdx.x >> 1, dir = blockIdx.x & 1;
  const double* D = bf + dir * part + (size_t)blk * 4096;
  for (int e = threadIdx.x; e < gbk::kTriTile; e += 256) {
    const gbk::TriEntry t = gbk::tri_entry(dir == 0, e & 31, e >> 5);
    out[(size_t)blockIdx.x * gbk::kTriTile + e] = D[t.k * 64 + t.row];
  }
}

cudaError_t form_on_device(const gbk::DevMat& d, size_t nnzb, const FactorTiles& ft, cudaStream_t s) {
  auto split = [&](const double* v, size_t n, const float* hi, const float* lo) {
    const unsigned blocks = (unsigned)std::min<size_t>((n + 255) / 256, 152 * 8);
    split_kernel<<<blocks, 256, 0, s>>>(v, n, const_cast<float*>(hi), const_cast<float*>(lo));
  };
  split(d.hb, nnzb * 16, d.hb_hi, d.hb_lo);
  split(d.sb, nnzb * 16, d.sb_hi, d.sb_lo);
  split(d.minv, (size_t)d.nb * 16, d.minv32, nullptr);
  diag_kernel<<<(d.n + 255) / 256, 256, 0, s>>>(d, const_cast<float*>(d.h_diag));
  if (d.bf_nblk > 0) {
    TileArgs t{};
    t.bf = d.bf64;
    t.part = (size_t)d.bf_nblk * 4096;
    t.n = d.n;
    t.bw = d.bf_bw;
    t.ne = ft.ne;
    for (int q = 0; q < 2; ++q) {
      t.sd[q] = std::ldexp(1.f, 4 - ft.ex[2 * q]);
      t.se[q] = std::ldexp(1.f, 4 - ft.ex[2 * q + 1]);
    }
    t.fx = reinterpret_cast<uint32_t*>(const_cast<uint4*>(d.fx));
    t.tf = const_cast<float*>(d.bfm);
    tile_kernel<<<2 * d.bf_nblk, 256, 0, s>>>(t);
    tri_pack_kernel<<<2 * d.bf_nblk, 256, 0, s>>>(d.bf64, t.part, const_cast<double*>(d.bft));
  }
  return cudaGetLastError();
}

// The dense inverse of S (dense_inverse.cuh) is kept for matrices without a banded
// factor of up to kDenseMax orbitals.  Solves gain beyond that too (1710 orbitals: 1944
// -> 860 ms), but every matrix pays for forming it, 4 n^2 bytes and O(n^3) FP64 work, used
// or not: at 1024 orbitals that is 4 MB and a few milliseconds, near what the rest of
// building the matrix takes.
constexpr int kDenseMax = 1024;
bool dense_wanted(int64_t n, bool factor) { return !factor && n <= kDenseMax; }

// Forms d.di; leaves it null where S is not SPD, the scratch cannot be had, or S is badly
// scaled or conditioned (the solves then iterate, and report such an S as before).  An FP32
// solve is accurate to some 1e-6 of the solution's largest entry, so a refinement level
// shrinks the residual by 1e-6 max |S| max |S^-1| and a few: 64 leaves 1e-4 (bundles: the
// product is 1.02).  s_max: max |S|.
constexpr double kDenseCond = 64.0;
cudaError_t form_dense_inverse(gbk::DevMat& d, uint4* frags, double s_max, cudaStream_t s) {
  const int np = (d.n + gbk::kDiB - 1) / gbk::kDiB * gbk::kDiB, nblk = np / gbk::kDiB, nt = (4 * d.nb + 15) / 16;
  const size_t one = sizeof(double) * (size_t)np * np, piv = sizeof(double) * gbk::kDiB * np;
  char* tmp = nullptr;
  if (cudaMalloc(&tmp, 2 * one + piv + 16) != cudaSuccess) {
    cudaGetLastError();
    return cudaSuccess;
  }
  double *A = reinterpret_cast<double*>(tmp), *B = reinterpret_cast<double*>(tmp + one);
  double* R = reinterpret_cast<double*>(tmp + 2 * one);
  auto* top = reinterpret_cast<unsigned long long*>(tmp + 2 * one + piv);
  int* bad = reinterpret_cast<int*>(top + 1);
  struct {
    unsigned long long top;
    int bad, pad;
  } h{};
  cudaError_t e = cudaMemsetAsync(top, 0, 16, s);
  if (e == cudaSuccess) {
    gbk::di_fill_kernel<<<np / 8, 256, 0, s>>>(d, A, np);
    for (int k = 0; k < nblk; ++k) {
      gbk::di_pivot_kernel<<<nblk, 256, 0, s>>>(A, np, k, R, bad);
      gbk::di_step_kernel<<<dim3(nblk, nblk), 256, 0, s>>>(A, B, np, k, R);
      std::swap(A, B);
    }
    gbk::di_max_kernel<<<152, 256, 0, s>>>(A, np, d.n, top);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, top, 16, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  double mx;
  std::memcpy(&mx, &h.top, sizeof mx);
  if (e == cudaSuccess && !h.bad && std::isfinite(mx) && mx > 0.0 && mx * s_max <= kDenseCond) {
    int ex;
    std::frexp(mx, &ex);
    if (ex > -40 && ex < 40) {  // largest entry in [2^14, 2^15)
      gbk::di_frag_kernel<<<dim3(nt, nt), 128, 0, s>>>(A, np, d.n, nt, std::ldexp(1.0, 15 - ex),
                                                        reinterpret_cast<uint32_t*>(frags));
      e = cudaGetLastError();
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      d.di = frags;
      d.di_nt = nt;
      d.di_ex = ex - 15;
    }
  }
  cudaFree(tmp);
  return e;
}

}  // namespace

extern "C" {

int32_t gb_abi_version(void) { return GB_ABI_VERSION; }

const char* gb_last_error(void) { return gb::g_err; }

gb_status gb_bsr_to_host(int64_t n, const int64_t* row_ptr, const int32_t* col_idx, const double* h_val,
                         const double* s_val, int64_t* nb, int64_t* nnzb, int32_t* blk_ptr, int32_t* blk_col,
                         double* blk_h, double* blk_s) {
  clear_error();
  if (!nb || !nnzb) return fail(GB_EINVAL, "nb and nnzb must not be NULL");
  HostBSR hb;
  gb_status st = build_host_bsr(n, row_ptr, col_idx, h_val, s_val, &hb);
  if (st != GB_OK) return st;
  *nb = hb.nb;
  *nnzb = hb.nnzb;
  if (blk_ptr) std::memcpy(blk_ptr, hb.blk_ptr.data(), sizeof(int32_t) * hb.blk_ptr.size());
  if (blk_col) std::memcpy(blk_col, hb.blk_col.data(), sizeof(int32_t) * hb.blk_col.size());
  if (blk_h) std::memcpy(blk_h, hb.blk_h.data(), sizeof(double) * hb.blk_h.size());
  if (blk_s) std::memcpy(blk_s, hb.blk_s.data(), sizeof(double) * hb.blk_s.size());
  return GB_OK;
}

gb_status gb_block_factor_to_host(int64_t n, const int64_t* row_ptr, const int32_t* col_idx, const double* h_val,
                                  const double* s_val, int32_t* bw, int64_t* nblk, double* factor) {
  clear_error();
  if (!bw || !nblk) return fail(GB_EINVAL, "bw and nblk must not be NULL");
  HostBSR hb;
  gb_status st = build_host_bsr(n, row_ptr, col_idx, h_val, s_val, &hb);
  if (st != GB_OK) return st;
  block_factor(&hb);
  *bw = hb.bf_bw;
  *nblk = hb.bf_nblk;
  if (factor && !hb.bf.empty()) std::memcpy(factor, hb.bf.data(), sizeof(double) * hb.bf.size());
  return GB_OK;
}

gb_status gb_build_bsr(int64_t n, const int64_t* row_ptr, const int32_t* col_idx, const double* h_val,
                       const double* s_val, void* stream, gb_matrix** out) {
  clear_error();
  if (!out) return fail(GB_EINVAL, "out must not be NULL");
  *out = nullptr;
  HostBSR hb;
  gb_status st = build_host_bsr(n, row_ptr, col_idx, h_val, s_val, &hb);
  if (st != GB_OK) return st;
  preconditioned_s_bounds(&hb);
  block_factor(&hb);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int dev = 0;
  GB_CUDA(cudaGetDevice(&dev));

  const size_t nnzb = hb.nnzb, nbl = hb.nb, nnz = hb.nnz;
  // one allocation, 256-byte aligned pieces
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = align256(off + bytes);
    return o;
  };
  const size_t o_bp = take(sizeof(int) * (nbl + 1)), o_bc = take(sizeof(int) * nnzb);
  const size_t o_hb = take(sizeof(double) * nnzb * 16), o_sb = take(sizeof(double) * nnzb * 16);
  const size_t o_mi = take(sizeof(double) * nbl * 16);
  const size_t o_rp = take(sizeof(int) * (n + 1)), o_ci = take(sizeof(int) * nnz);
  const size_t o_hv = take(sizeof(double) * nnz), o_sv = take(sizeof(double) * nnz);
  const size_t nbf = hb.bf.size();  // 4 x nblk x 4096 factor entries (0: no factor)
  const FactorTiles ft = factor_tiles(hb);
  const size_t nblk = nbf ? (size_t)hb.bf_nblk : 0;
  const size_t o_bf64 = take(sizeof(double) * nbf);
  const size_t up = off;  // uploaded; the rest is formed from it on the device
  const size_t o_hh = take(sizeof(float) * nnzb * 16), o_hl = take(sizeof(float) * nnzb * 16);
  const size_t o_sh = take(sizeof(float) * nnzb * 16), o_sl = take(sizeof(float) * nnzb * 16);
  const size_t o_m32 = take(sizeof(float) * nbl * 16), o_hd = take(sizeof(float) * n);
  const size_t o_bfm = take(sizeof(float) * 2 * nblk * gbk::kMmaTileFloatsDev);
  const size_t o_bft = take(sizeof(double) * 2 * nblk * gbk::kTriTile);
  const size_t o_fx = take(ft.ok ? sizeof(uint4) * 2 * nblk * gbk::fx_block_words(ft.ne) : 0);
  const bool dense = dense_wanted(n, nbf != 0);
  const size_t dnt = dense ? (4 * nbl + 15) / 16 : 0;
  const size_t o_di = take(sizeof(uint4) * 64 * dnt * dnt);
  const size_t total = off;

  std::unique_ptr<char[]> host(new char[up]);
  auto put = [&](size_t o, const void* src, size_t bytes) { std::memcpy(host.get() + o, src, bytes); };
  put(o_bp, hb.blk_ptr.data(), sizeof(int) * (nbl + 1));
  put(o_bc, hb.blk_col.data(), sizeof(int) * nnzb);
  put(o_hb, hb.blk_h.data(), sizeof(double) * nnzb * 16);
  put(o_sb, hb.blk_s.data(), sizeof(double) * nnzb * 16);
  put(o_mi, hb.minv.data(), sizeof(double) * nbl * 16);
  {
    int* rp = reinterpret_cast<int*>(host.get() + o_rp);
    for (int64_t i = 0; i <= n; ++i) rp[i] = (int)hb.row_ptr[i];
  }
  put(o_ci, hb.col_idx.data(), sizeof(int) * nnz);
  put(o_hv, hb.h_val.data(), sizeof(double) * nnz);
  put(o_sv, hb.s_val.data(), sizeof(double) * nnz);
  if (nbf) put(o_bf64, hb.bf.data(), sizeof(double) * nbf);

  gb_matrix* m = new gb_matrix();
  m->device = dev;
  m->n = n;
  m->nb = hb.nb;
  m->nnz = hb.nnz;
  m->nnzb = hb.nnzb;
  m->max_row = hb.max_row;
  m->h_row_ptr = hb.row_ptr;
  cudaError_t e = cudaMalloc(&m->base, total);
  if (e != cudaSuccess) {
    delete m;
    return fail(GB_ENOMEM, "cudaMalloc(%zu bytes) for the matrix failed: %s", total, cudaGetErrorString(e));
  }
  char* b = static_cast<char*>(m->base);
  gbk::DevMat& d = m->dm;
  d.n = (int)n;
  d.nb = (int)hb.nb;
  d.blk_ptr = reinterpret_cast<const int*>(b + o_bp);
  d.blk_col = reinterpret_cast<const int*>(b + o_bc);
  d.hb = reinterpret_cast<const double*>(b + o_hb);
  d.sb = reinterpret_cast<const double*>(b + o_sb);
  d.hb_hi = reinterpret_cast<const float*>(b + o_hh);
  d.hb_lo = reinterpret_cast<const float*>(b + o_hl);
  d.sb_hi = reinterpret_cast<const float*>(b + o_sh);
  d.sb_lo = reinterpret_cast<const float*>(b + o_sl);
  d.minv = reinterpret_cast<const double*>(b + o_mi);
  d.minv32 = reinterpret_cast<const float*>(b + o_m32);
  d.row_ptr = reinterpret_cast<const int*>(b + o_rp);
  d.col_idx = reinterpret_cast<const int*>(b + o_ci);
  d.h_val = reinterpret_cast<const double*>(b + o_hv);
  d.s_val = reinterpret_cast<const double*>(b + o_sv);
  d.h_diag = reinterpret_cast<const float*>(b + o_hd);
  d.s_lam_min = hb.lam_min;
  d.s_lam_max = hb.lam_max;
  d.bf_bw = nbf ? hb.bf_bw : 0;
  d.bf_nblk = nbf ? (int)hb.bf_nblk : 0;
  d.bf64 = nbf ? reinterpret_cast<const double*>(b + o_bf64) : nullptr;
  d.bft = nbf ? reinterpret_cast<const double*>(b + o_bft) : nullptr;
  d.fx = ft.ok ? reinterpret_cast<const uint4*>(b + o_fx) : nullptr;
  d.fx_ne = ft.ne;
  d.fx_lg = ft.lg;
  for (int q = 0; q < 2; ++q) {
    d.fx_kd[q] = ft.kd[q];
    d.fx_ke[q] = ft.ke[q];
  }
  d.bfm = nbf ? reinterpret_cast<const float*>(b + o_bfm) : nullptr;
  e = cudaMemcpyAsync(m->base, host.get(), up, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = form_on_device(d, nnzb, ft, s);
  d.di = nullptr;
  if (e == cudaSuccess && dense) {
    double s_max = 0.0;
    for (double v : hb.s_val) s_max = std::max(s_max, std::fabs(v));
    e = form_dense_inverse(d, reinterpret_cast<uint4*>(b + o_di), s_max, s);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    cudaFree(m->base);
    delete m;
    return cuda_fail(e, "matrix upload");
  }
  *out = m;
  return GB_OK;
}

gb_status gb_matrix_get_info(const gb_matrix* m, gb_matrix_info* info) {
  clear_error();
  if (!m || !info) return fail(GB_EINVAL, "NULL argument");
  info->n = m->n;
  info->nnz = m->nnz;
  info->nb = m->nb;
  info->nnzb = m->nnzb;
  info->max_row = m->max_row;
  info->block = 4;
  info->device = m->device;
  info->factor_bw = m->dm.bf_bw;
  info->s_lam_min = m->dm.s_lam_min;
  info->s_lam_max = m->dm.s_lam_max;
  info->factor_nblk = m->dm.bf_nblk;
  return GB_OK;
}

void gb_free(gb_matrix* m) {
  if (!m) return;
  if (m->base) {
    cudaDeviceSynchronize();
    cudaFree(m->base);
  }
  delete m;
}

gb_status gb_spmm(const gb_matrix* m, int32_t which, gb_precision prec, int32_t w, const void* x, void* y,
                  void* stream) {
  clear_error();
  if (!m || !x || !y) return fail(GB_EINVAL, "NULL argument");
  if (which != 0 && which != 1) return fail(GB_EINVAL, "which must be 0 (H) or 1 (S)");
  if (w < 1 || w > 64) return fail(GB_EINVAL, "w must be in [1, 64]");
  if (prec != GB_FP64 && prec != GB_MIXED) return fail(GB_EINVAL, "bad precision");
  if (misaligned(x, prec == GB_FP64 ? 16 : 8) || misaligned(y, prec == GB_FP64 ? 16 : 8))
    return fail(GB_EINVAL, "x and y must be aligned to their complex element (16 bytes FP64, 8 FP32)");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const long long outs = (long long)m->n * w;
  auto blocks = [](long long threads) { return (unsigned)((threads + 255) / 256); };
  if (prec == GB_FP64) {
    const double* A = which ? m->dm.s_val : m->dm.h_val;
    const auto* xd = static_cast<const double2*>(x);
    auto* yd = static_cast<double2*>(y);
    if (w == 1)
      spmm_csr_d_kernel<4><<<blocks(4 * outs), 256, 0, s>>>(m->dm, A, w, xd, yd);
    else if (w == 2)
      spmm_csr_d_kernel<2><<<blocks(2 * outs), 256, 0, s>>>(m->dm, A, w, xd, yd);
    else
      spmm_csr_d_kernel<1><<<blocks(outs), 256, 0, s>>>(m->dm, A, w, xd, yd);
  } else {
    const float* A = which ? m->dm.sb_hi : m->dm.hb_hi;
    const auto* x2 = static_cast<const float2*>(x);
    const auto* x4 = static_cast<const float4*>(x);
    auto* y2 = static_cast<float2*>(y);
    auto* y4 = static_cast<float4*>(y);
    const bool aligned = (reinterpret_cast<uintptr_t>(x) % 16) == 0 && (reinterpret_cast<uintptr_t>(y) % 16) == 0;
    const unsigned wb = (unsigned)((m->nb + 7) / 8);  // 8 warps = 8 block rows per CTA
    auto run = [&](auto rag) {
      constexpr bool RAG = decltype(rag)::value;
      switch (aligned || w <= 2 ? w : 0) {
        case 1:
          if (aligned)
            spmm_quad_kernel<1, RAG><<<wb, 256, 0, s>>>(m->dm, A, x2, y2);
          else
            spmm_quad_kernel<1, RAG, true><<<wb, 256, 0, s>>>(m->dm, A, x2, y2);
          break;
        case 2:
          if (aligned)
            spmm_quad_kernel<2, RAG><<<wb, 256, 0, s>>>(m->dm, A, x2, y2);
          else
            spmm_quad_kernel<2, RAG, true><<<wb, 256, 0, s>>>(m->dm, A, x2, y2);
          break;
        case 4: spmm_wide_kernel<2, RAG><<<wb, 256, 0, s>>>(m->dm, A, x4, y4); break;
        case 8: spmm_wide_kernel<4, RAG><<<wb, 256, 0, s>>>(m->dm, A, x4, y4); break;
        case 16: spmm_wide_kernel<8, RAG><<<wb, 256, 0, s>>>(m->dm, A, x4, y4); break;
        case 32: spmm_wide_kernel<16, RAG><<<wb, 256, 0, s>>>(m->dm, A, x4, y4); break;
        case 64: spmm_wide_kernel<32, RAG><<<wb, 256, 0, s>>>(m->dm, A, x4, y4); break;
        default:
          spmm_any_kernel<RAG><<<blocks(w <= 8 ? 32 * m->nb : m->nb * w), 256, 0, s>>>(m->dm, A, w, x2, y2);
      }
    };
    if (m->n % 4 != 0)
      run(std::true_type{});
    else
      run(std::false_type{});
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "spmm launch");
  return GB_OK;
}

}  // extern "C"

// ------------------------------------------------------------ shifted solve
namespace {

// Inner solver: the exact block-bidiagonal Cholesky solve when S's
// half-bandwidth is at most 63 (both precisions), unless flags ask for an
// iteration.  Otherwise the mixed path runs Chebyshev when the spectrum bounds
// of the preconditioned S are known and positive (CG with flags bit 2), and
// the FP64 path runs CG.  K Chebyshev steps reduce the preconditioned residual
// below itol by the bound 2 sqrt(kappa) q^K (q = (sqrt(kappa) - 1) /
// (sqrt(kappa) + 1)), with the Lanczos bounds widened by 2% on each side.
constexpr int kFlagSmem = 2, kFlagCG = 4, kFlagCheb = 16, kFlagHpF32 = 32, kFlagStall = 64;
constexpr int kStallWindow = 3000;  // iterations without halving the best residual
// Without a factor the mixed path's real recurrence takes the dense inverse where
// the matrix keeps one, unless flags ask for an iteration or its shared-memory vectors.
bool dense_inner(const gb_matrix* m, const gb_solve_params* p, bool real) {
  return m->dm.di && real && p->prec == GB_MIXED && !(p->flags & (kFlagCG | kFlagCheb | kFlagSmem));
}
// Refinement levels of the FP32 solves: two for tol >= 1e-6, three down to 1e-9, four
// below (at tol 1e-10 a near-threshold pair of a 114-orbital chain stagnated at 7.7e-10
// with three levels and converged with four).  An explicit bound on the application's
// error asks for (2e-6)^levels <= bound, two at least (2e-6: the measured accuracy of
// one FP32 factor solve).
int refinement_levels(double tol, double bound) {
  if (!(bound > 0)) return tol >= 1e-6 ? 2 : (tol >= 1e-9 ? 3 : 4);
  int l = 2;
  while (l < 4 && std::pow(2e-6, l) > bound) ++l;
  return l;
}
void set_inner_method(const gb_matrix* m, const gb_solve_params* p, double itol, bool real, gbk::Args& a) {
  std::memset(&a, 0, sizeof a);
  a.hp_fp32 = (p->prec == GB_MIXED && (p->flags & kFlagHpF32)) ? 1 : 0;
  a.stall = (p->flags & kFlagStall) ? kStallWindow : 0;
  if (!(p->flags & (kFlagCG | kFlagCheb)) && m->dm.bf_bw > 0) {
    a.inner_bchol = 1;  // exact: block-bidiagonal Cholesky factor solves
    a.bc_levels = refinement_levels(p->tol, p->inner_tol);
    return;
  }
  if (dense_inner(m, p, real)) {
    // an iteration's inner_tol (1e-7 by default) holds per level, of which there are two:
    // an application's error stays below its square
    a.inner_dense = 1;
    a.bc_levels = p->inner_tol > 0 ? refinement_levels(p->tol, p->inner_tol * p->inner_tol)
                                   : std::max(3, refinement_levels(p->tol, 0.0));
    return;
  }
  const double lmin = m->dm.s_lam_min * 0.98, lmax = m->dm.s_lam_max * 1.02;
  if (p->prec != GB_MIXED || (p->flags & kFlagCG) || !(lmin > 0.0) || !(lmax > lmin)) return;
  const double kappa = lmax / lmin, sk = std::sqrt(kappa);
  const double q = (sk - 1.0) / (sk + 1.0);
  int K = (int)std::ceil(std::log(2.0 * sk / itol) / std::log(1.0 / q));
  K = std::max(1, std::min(K, 48));
  const double theta = 0.5 * (lmax + lmin), delta = 0.5 * (lmax - lmin), sigma = theta / delta;
  double rho = 1.0 / sigma;
  for (int k = 0; k < K; ++k) {
    const double rn = 1.0 / (2.0 * sigma - rho);
    a.cheb_A[k] = (float)(rn * rho);
    a.cheb_B[k] = (float)(2.0 * rn / delta);
    rho = rn;
  }
  a.cheb_c0 = (float)(1.0 / theta);
  a.cheb_K = K;
  a.inner_cheb = 1;
}

// Which recurrence solves the panels.  The real three-term recurrence
// (panel_real.cuh) does, except where the caller names a seed shift or asks for
// panels of one or two columns, and in the mixed path where S's factor does not fit
// the FP16 tiles (factor_tiles): those run the seed recurrence (panel.cuh), whose
// TF32 tiles keep an exponent per entry.  The FP64 correction of stagnating columns
// is built on it (one-column panels, another seed each time).
bool real_recurrence(const gb_matrix* m, const gb_solve_params* p) {
  const bool factor = m->dm.bf_bw > 0 && !(p->flags & (kFlagCG | kFlagCheb));
  if (p->prec == GB_MIXED && factor && !m->dm.fx) return false;
  return p->seed_shift < 0 && p->panel != 1 && p->panel != 2;
}

// Team-workspace layout of panels of W pairs (real recurrence) or W complex
// columns (seed recurrence).
size_t layout_team(size_t N4, int W, int K, int KG, int maxit, int Mcap, bool want_g, bool real, gbk::Args& a) {
  const size_t Kz = K, R = real ? 2 * (size_t)W : W, mx = maxit;
  const size_t esz = real ? 8 : 16;  // a history entry: v is real, r complex
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = align256(off + bytes);
    return o;
  };
  const size_t vec = N4 * W * 16;
  a.o_r = take(vec);
  a.o_rt = take(vec);
  a.o_p = real ? 0 : take(vec);
  a.o_sp = real ? 0 : take(vec);
  a.o_u = take(vec);
  a.o_w = take(vec);
  a.o_g = take(vec);
  a.o_d = take(vec);
  a.o_q = take(vec);
  a.o_x = take(vec);
  a.o_hr = take((mx + 1) * (size_t)Mcap * esz);
  a.o_ab = take(mx * R * (real ? 24 : 32));
  a.o_L = real ? 0 : take((mx + 1) * R * sizeof(int));
  a.o_t = take((mx + 1) * R * esz);
  a.o_ck = take((mx / gbk::CK + 1) * R * Kz * 2 * 16);
  a.o_pi = take(R * Kz * 2 * 16);
  a.o_nk = take(R * Kz * sizeof(int));
  a.o_res = take(R * Kz * sizeof(double));
  a.o_buf = take((gbk::CK + 1) * R * Kz * 16);
  a.o_cp = take((mx + 1) * R * KG * 2 * esz);
  a.o_cf = take((mx + 1) * R * 2 * esz);
  a.o_cg = want_g ? take((mx + 1) * R * Kz * 16) : 0;
  return off;
}

const void* team_fn(bool fp64, bool real) {
  if (real) return fp64 ? (const void*)gbk::team_kernel<false, true> : (const void*)gbk::team_kernel<true, true>;
  return fp64 ? (const void*)gbk::team_kernel<false, false> : (const void*)gbk::team_kernel<true, false>;
}
const void* batched_fn(bool fp64, bool real) {
  if (real)
    return fp64 ? (const void*)gbk::team_kernel_batched<false, true> : (const void*)gbk::team_kernel_batched<true, true>;
  return fp64 ? (const void*)gbk::team_kernel_batched<false, false> : (const void*)gbk::team_kernel_batched<true, false>;
}
gb_status launch_team(gbk::Args& a, bool fp64, bool real, int teams, int threads, size_t dyn, cudaStream_t s) {
  const void* fn = team_fn(fp64, real);
  GB_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
  void* args[] = {&a};
  GB_CUDA(cudaLaunchKernel(fn, dim3(teams), dim3(threads), args, dyn, s));
  return GB_OK;
}

struct Plan {
  int C;  // right-hand sides per panel
  int threads;
  bool real;
  int W, KG, npanels, teams, teams_per_sm, Mcap, inner_maxit, cg_smem;
  size_t dyn_smem;
  double itol;
  size_t team_bytes, header_bytes, total;
  size_t o_z, o_wr, o_we, o_cols, o_off, o_status, o_counter;
  gbk::Args a;
};

// full_hist: the plan of a verification run; recurrence: 0 the seed's, 1 the real one, else
// real_recurrence's choice
gb_status make_plan(const gb_matrix* m, const gb_solve_params* p, bool want_g, Plan* pl, bool full_hist = false,
                    int recurrence = -1) {
  if (!m) return fail(GB_EINVAL, "matrix is NULL");
  if (!p) return fail(GB_EINVAL, "params is NULL");
  if (p->nshift < 1 || p->nshift > 256) return fail(GB_EINVAL, "nshift must be in [1, 256]");
  if (!p->z_re || !p->z_im) return fail(GB_EINVAL, "shift arrays are NULL");
  for (int k = 0; k < p->nshift; ++k)
    if (!std::isfinite(p->z_re[k]) || !std::isfinite(p->z_im[k]) || !(p->z_im[k] > 0.0))
      return fail(GB_EINVAL, "shift %d must be finite with Im z > 0", k);
  if (p->nrhs < 1 || !p->rhs_cols) return fail(GB_EINVAL, "need nrhs >= 1 and rhs_cols");
  for (int i = 0; i < p->nrhs; ++i)
    if (p->rhs_cols[i] < 0 || p->rhs_cols[i] >= m->n) return fail(GB_EINVAL, "rhs_cols[%d] out of range", i);
  if (!(p->tol > 0.0) || !std::isfinite(p->tol)) return fail(GB_EINVAL, "tol must be > 0");
  if (p->maxit < 1 || p->maxit > 1000000) return fail(GB_EINVAL, "maxit must be in [1, 1e6]");
  if (p->prec != GB_FP64 && p->prec != GB_MIXED) return fail(GB_EINVAL, "bad precision");
  if (p->seed_shift >= p->nshift) return fail(GB_EINVAL, "seed_shift out of range");
  const double* ws[2] = {p->w_rho, p->w_edm};
  for (int q = 0; q < 2; ++q)
    if (ws[q])
      for (int k = 0; k < 2 * p->nshift; ++k)
        if (!std::isfinite(ws[q][k])) return fail(GB_EINVAL, "non-finite quadrature weight");

  cudaDeviceProp prop;
  cudaError_t e = cudaGetDeviceProperties(&prop, m->device);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDeviceProperties");
  const int nsm = prop.multiProcessorCount;

  // Panel width W and inner-CG placement.  The inner-CG vectors g, d, q of a
  // panel (3 x N4 x W elements) may live in shared memory (flag bit 1) when
  // they fit; by default they stay in global memory so that several teams
  // share each SM.  Auto W: the widest panel that still gives every resident
  // team a panel.
  const size_t n4 = 4 * (size_t)m->nb;
  const size_t cg_esz = p->prec == GB_FP64 ? 16 : 8;
  const size_t smem_budget = (size_t)prop.sharedMemPerBlockOptin - 40 * 1024;
  // the exact factor solve keeps its partial sums, its current block and (FP32)
  // two staged factor tiles in dynamic shared memory instead
  const bool bchol = !(p->flags & (kFlagCG | kFlagCheb)) && m->dm.bf_bw > 0;
  const bool want_smem = (p->flags & kFlagSmem) != 0 && !bchol;
  const bool f64 = p->prec == GB_FP64, real = recurrence < 0 ? real_recurrence(m, p) : recurrence != 0;
  auto width = [&](int cols) { return real ? std::max(1, cols / 2) : cols; };  // stored pairs or complex columns
  auto fits = [&](int w) { return want_smem && 3 * n4 * (size_t)w * cg_esz + gbk::kRedBytes <= smem_budget; };
  auto dyn_bytes = [&](int w) -> size_t {
    const unsigned cg = fits(w) ? (unsigned)(3 * n4 * (size_t)w * cg_esz) : 0u;
    return gbk::dyn_layout(f64, w, bchol, cg, m->dm.bf_bw, !real).bytes;
  };
  auto occupancy = [&](size_t dyn) {
    int per_sm = 1;
    const void* fn = team_fn(f64, real);
    if (dyn > 0) cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    const cudaError_t oe = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, gbk::TPB, dyn);
    return (oe != cudaSuccess || per_sm < 1) ? 1 : per_sm;
  };
  int C = p->panel;
  if (C <= 0) {
    // one wave that fills >= 3/4 of the team slots beats 1.5 waves of half-size
    // panels (measured on the 1900-orbital chain: 8 columns, 238 panels on 304
    // slots, ~20% faster than 4)
    C = 1;
    if (real && !f64) {
      // one wide team per SM: the narrowest panels that fit one wave (912
      // orbitals, all columns: 8 columns 275 us an iteration, 4 columns two teams
      // per SM 325, 16 columns 427; 1900 orbitals: 16 columns 490, 8 columns 502)
      C = 2;
      while (C < 32 && (p->nrhs + C - 1) / C > nsm) C *= 2;
    }
    if (C == 1 || (p->nrhs + C - 1) / C > nsm) {
      // two teams per SM: one wave that fills >= 3/4 of the team slots beats 1.5
      // waves of half-size panels
      C = 1;
      for (int cand : {32, 16, 8, 4, 2}) {
        const size_t dyn = dyn_bytes(width(cand));
        if (4LL * ((p->nrhs + cand - 1) / cand) >= 3LL * nsm * occupancy(dyn)) {
          C = cand;
          break;
        }
      }
    }
    if (real && C == 1 && p->nrhs > 1) C = 2;  // a pair costs what one of its columns does
  }
  if (C != 1 && C != 2 && C != 4 && C != 8 && C != 16 && C != 32)
    return fail(GB_EINVAL, "panel must be 1, 2, 4, 8, 16 or 32");
  const int W = width(C);
  pl->C = C;
  pl->real = real;
  pl->W = W;
  pl->cg_smem = fits(W) ? 1 : 0;
  pl->dyn_smem = dyn_bytes(W);
  pl->teams_per_sm = occupancy(pl->dyn_smem);
  pl->KG = (p->nshift + 31) / 32;
  pl->npanels = (p->nrhs + C - 1) / C;
  pl->teams = std::min(pl->npanels, nsm * pl->teams_per_sm);
  // one wide team per SM where the launch would leave SMs with a single team
  pl->threads = real && !f64 && pl->npanels <= nsm ? gbk::TPB_WIDE : gbk::TPB;
  pl->Mcap = full_hist ? (real ? 2 * W : W) * 4 * (int)m->nb : C * m->max_row;
  pl->inner_maxit = 500;
  // Inner-solve accuracy: the seed recurrence treats w = S^{-1} H p as exact,
  // and each iteration's error enters the shifted residual gap, so the inner
  // solve runs close to working precision (FP64: 1e-14; mixed: 1e-7 per FP32
  // refinement level, ~1e-14 after the float-float residual step).
  if (p->prec == GB_FP64)
    pl->itol = p->inner_tol > 0 ? p->inner_tol : 1e-14;
  else
    pl->itol = p->inner_tol > 0 ? p->inner_tol : 1e-7;

  set_inner_method(m, p, pl->itol, real, pl->a);
  pl->a.bc_bw_alloc = m->dm.bf_bw;
  const size_t K = p->nshift, N4 = 4 * (size_t)m->nb;
  pl->team_bytes = layout_team(N4, W, (int)K, pl->KG, p->maxit, pl->Mcap, want_g, real, pl->a);
  pl->a.C = C;

  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = align256(off + bytes);
    return o;
  };
  pl->o_z = take(K * 16);
  pl->o_wr = take(K * 16);
  pl->o_we = take(K * 16);
  pl->o_cols = take(sizeof(int) * p->nrhs);
  pl->o_off = take(sizeof(long long) * (p->nrhs + 1));
  pl->o_status = take(sizeof(int) * p->nrhs);
  pl->o_counter = take(sizeof(int));
  pl->header_bytes = off;
  pl->total = pl->header_bytes + pl->team_bytes * pl->teams + 256;
  return GB_OK;
}

}  // namespace

extern "C" {

gb_status gb_solve_plan(const gb_matrix* m, const gb_solve_params* p, int32_t* plan) {
  clear_error();
  if (!plan) return fail(GB_EINVAL, "plan is NULL");
  Plan pl;
  gb_status st = make_plan(m, p, false, &pl);
  if (st != GB_OK) return st;
  plan[0] = pl.C;
  plan[1] = pl.teams;
  plan[2] = pl.cg_smem;
  plan[3] = (int32_t)pl.dyn_smem;
  plan[4] = pl.a.inner_dense ? 3 : (pl.a.inner_bchol ? 2 : (pl.a.inner_cheb ? 1 : 0));
  plan[5] = pl.teams_per_sm;
  return GB_OK;
}

size_t gb_solve_workspace_size(const gb_matrix* m, const gb_solve_params* p) {
  clear_error();
  Plan pl;
  if (make_plan(m, p, true, &pl) != GB_OK) return 0;
  return pl.total;
}

gb_status gb_shifted_solve(const gb_matrix* m, const gb_solve_params* p, const gb_outputs* out, void* workspace,
                           size_t workspace_bytes, void* stream) {
  clear_error();
  if (!out) return fail(GB_EINVAL, "outputs is NULL");
  if (check_outputs(out) != GB_OK) return GB_EINVAL;
  Plan pl;
  const bool want_g = out->g_proj != nullptr;
  gb_status st = make_plan(m, p, want_g, &pl);
  if (st != GB_OK) return st;
  if (!workspace) return fail(GB_EINVAL, "workspace is NULL");
  if ((reinterpret_cast<uintptr_t>(workspace) & 255) != 0) return fail(GB_EINVAL, "workspace must be 256-byte aligned");
  if (workspace_bytes < pl.total)
    return fail(GB_ENOMEM, "workspace too small: %zu < %zu bytes", workspace_bytes, pl.total);
  int dev = 0;
  GB_CUDA(cudaGetDevice(&dev));
  if (dev != m->device) return fail(GB_EINVAL, "current device %d differs from the matrix's device %d", dev, m->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);

  const int K = p->nshift, nrhs = p->nrhs;
  // packed output offsets: prefix sums of |R_j|
  std::vector<char> hdr(pl.header_bytes, 0);
  double2* hz = reinterpret_cast<double2*>(hdr.data() + pl.o_z);
  double2* hwr = reinterpret_cast<double2*>(hdr.data() + pl.o_wr);
  double2* hwe = reinterpret_cast<double2*>(hdr.data() + pl.o_we);
  for (int k = 0; k < K; ++k) {
    hz[k] = make_double2(p->z_re[k], p->z_im[k]);
    hwr[k] = p->w_rho ? make_double2(p->w_rho[2 * k], p->w_rho[2 * k + 1]) : make_double2(0, 0);
    hwe[k] = p->w_edm ? make_double2(p->w_edm[2 * k], p->w_edm[2 * k + 1]) : make_double2(0, 0);
  }
  std::memcpy(hdr.data() + pl.o_cols, p->rhs_cols, sizeof(int) * nrhs);
  const std::vector<int64_t>& rp = m->h_row_ptr;
  long long* ho = reinterpret_cast<long long*>(hdr.data() + pl.o_off);
  ho[0] = 0;
  for (int i = 0; i < nrhs; ++i) {
    const int j = p->rhs_cols[i];
    ho[i + 1] = ho[i] + (rp[j + 1] - rp[j]);
  }
  char* wsb = static_cast<char*>(workspace);
  GB_CUDA(cudaMemcpyAsync(wsb, hdr.data(), pl.header_bytes, cudaMemcpyHostToDevice, s));

  gbk::Args& a = pl.a;
  a.m = m->dm;
  a.K = K;
  a.W = pl.W;
  a.KG = pl.KG;
  a.nrhs = nrhs;
  a.npanels = pl.npanels;
  a.maxit = p->maxit;
  a.inner_maxit = pl.inner_maxit;
  a.has_rho = p->w_rho != nullptr;
  a.has_edm = p->w_edm != nullptr;
  a.want_g = want_g;
  a.tol = p->tol;
  a.itol = pl.itol;
  const int seed = p->seed_shift >= 0 ? p->seed_shift : K / 2;
  a.sigma = make_double2(p->z_re[seed], p->z_im[seed]);
  a.z = reinterpret_cast<const double2*>(wsb + pl.o_z);
  a.w_rho = reinterpret_cast<const double2*>(wsb + pl.o_wr);
  a.w_edm = reinterpret_cast<const double2*>(wsb + pl.o_we);
  a.rhs_cols = reinterpret_cast<const int*>(wsb + pl.o_cols);
  a.out_off = reinterpret_cast<const long long*>(wsb + pl.o_off);
  a.status = reinterpret_cast<int*>(wsb + pl.o_status);
  a.panel_counter = reinterpret_cast<int*>(wsb + pl.o_counter);
  a.team_ws = wsb + align256(pl.header_bytes);
  a.team_bytes = pl.team_bytes;
  a.Mcap = pl.Mcap;
  a.ldos = out->ldos;
  a.rho = out->rho;
  a.edm = out->edm;
  a.q = out->q;
  a.e_loc = out->e_loc;
  a.iters = out->iters;
  a.inner_iters = out->inner_iters;
  a.col_status = out->col_status;
  a.conv = out->converged;
  a.resid = out->resid;
  a.g_proj = reinterpret_cast<double2*>(out->g_proj);
  a.P = ho[nrhs];

  a.cg_smem = pl.cg_smem;
  if ((st = launch_team(a, p->prec == GB_FP64, pl.real, pl.teams, pl.threads, pl.dyn_smem, s)) != GB_OK) return st;
  std::vector<int> hst(nrhs);
  GB_CUDA(cudaMemcpyAsync(hst.data(), a.status, sizeof(int) * nrhs, cudaMemcpyDeviceToHost, s));
  GB_CUDA(cudaStreamSynchronize(s));
  int any = 0;
  for (int v : hst) any |= v;
  if (any & gbk::kStTimeout) return fail(GB_ETIMEOUT, "a bounded wait for a staged factor tile gave up");
  if (any & gbk::kStNotSPD) return fail(GB_ENOTSPD, "inner CG found S not positive definite");
  if (any & gbk::kStBreakdown) return fail(GB_EBREAKDOWN, "COCG breakdown in at least one column");
  if (any & (gbk::kStNoConv | gbk::kStInner))
    return fail(GB_ENOCONV, "some (shift, column) pairs did not reach tol within maxit%s",
                (any & gbk::kStInner) ? " (inner CG hit its cap)" : "");
  return GB_OK;
}

}  // extern "C"

// ------------------------------------------------------------ standalone exact S^-1
// One team applies the block-bidiagonal Cholesky solve to a panel of W
// columns (the inner solve of the shifted recurrence, on its own: for tests
// and for timing the factor solve).
namespace {

template <typename T>
__global__ void __launch_bounds__(gbk::TPB, 1)
    sinv_kernel(const __grid_constant__ gbk::Args a, const typename gbk::CplxOf<T>::type* x,
                typename gbk::CplxOf<T>::type* y, typename gbk::CplxOf<T>::type* t1,
                typename gbk::CplxOf<T>::type* t2, int* status) {
  __shared__ gbk::Smem sm;
  extern __shared__ __align__(16) char dyn_smem[];
  gbk::team_init(sm, dyn_smem);
  if (threadIdx.x < gbk::WMAX) sm.act[threadIdx.x] = threadIdx.x < a.W ? 1 : 0;
  if (threadIdx.x == 0) sm.inner_count = 0;
  __syncthreads();
  if (sizeof(T) == 4 && !a.m.fx) {
    if constexpr (sizeof(T) == 4) gbk::seed_solve(a, sm, x, y, t1);
  } else if constexpr (sizeof(T) == 4) {
    float m0 = 0.f, m1 = 0.f;
    for (int e = threadIdx.x; e < 4 * a.m.nb * a.W; e += gbk::TPB) {
      m0 = fmaxf(m0, fabsf(x[e].x));
      m1 = fmaxf(m1, fabsf(x[e].y));
    }
    gbk::col_max(sm, a.W, m0, m1);
    __syncthreads();
    gbk::fx_solve<true>(a, sm, x, y, t1, t2);
  } else {
    gbk::bc_solve64(a, sm, x, y, t1, t2);
  }
  if (threadIdx.x == 0) *status = sm.bc_fail ? gbk::kStTimeout : 0;
}

}  // namespace

extern "C" {

gb_status gb_apply_sinv(const gb_matrix* m, gb_precision prec, int32_t w, const void* x, void* y, void* stream) {
  clear_error();
  if (!m || !x || !y) return fail(GB_EINVAL, "NULL argument");
  if (w != 1 && w != 2 && w != 4 && w != 8 && w != 16 && w != 32)
    return fail(GB_EINVAL, "w must be 1, 2, 4, 8, 16 or 32");
  if (prec != GB_FP64 && prec != GB_MIXED) return fail(GB_EINVAL, "bad precision");
  if (m->dm.bf_bw <= 0) return fail(GB_EINVAL, "no factor: S's half-bandwidth exceeds 63");
  if (misaligned(x, prec == GB_FP64 ? 16 : 8) || misaligned(y, prec == GB_FP64 ? 16 : 8))
    return fail(GB_EINVAL, "x and y must be aligned to their complex element");
  int dev = 0;
  GB_CUDA(cudaGetDevice(&dev));
  if (dev != m->device) return fail(GB_EINVAL, "current device %d differs from the matrix's device %d", dev, m->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool f64 = prec == GB_FP64;
  const size_t esz = f64 ? 16 : 8, n4 = 4 * (size_t)m->nb, panel = esz * n4 * w;
  // padded input, output and two scratch panels, plus the status word
  char* buf = nullptr;
  GB_CUDA(cudaMallocAsync(reinterpret_cast<void**>(&buf), 4 * panel + 256, s));
  char* xin = buf;
  char* yout = buf + panel;
  int* st = reinterpret_cast<int*>(buf + 4 * panel);
  cudaError_t e = cudaMemsetAsync(buf, 0, 4 * panel + 256, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(xin, x, esz * m->n * w, cudaMemcpyDeviceToDevice, s);
  gbk::Args a;
  std::memset(&a, 0, sizeof a);
  a.m = m->dm;
  a.W = w;
  a.inner_bchol = 1;
  a.bc_bw_alloc = m->dm.bf_bw;
  const size_t dyn = gbk::dyn_layout(f64, w, true, 0, m->dm.bf_bw, !m->dm.fx).bytes;
  if (e == cudaSuccess) {
    if (f64) {
      e = cudaFuncSetAttribute(sinv_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
      if (e == cudaSuccess)
        sinv_kernel<double><<<1, gbk::TPB, dyn, s>>>(a, reinterpret_cast<const double2*>(xin),
                                                      reinterpret_cast<double2*>(yout),
                                                      reinterpret_cast<double2*>(buf + 2 * panel),
                                                      reinterpret_cast<double2*>(buf + 3 * panel), st);
    } else {
      e = cudaFuncSetAttribute(sinv_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
      if (e == cudaSuccess)
        sinv_kernel<float><<<1, gbk::TPB, dyn, s>>>(a, reinterpret_cast<const float2*>(xin),
                                                    reinterpret_cast<float2*>(yout),
                                                    reinterpret_cast<float2*>(buf + 2 * panel),
                                                    reinterpret_cast<float2*>(buf + 3 * panel), st);
    }
    if (e == cudaSuccess) e = cudaGetLastError();
  }
  int hst = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(y, yout, esz * m->n * w, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hst, st, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFreeAsync(buf, s);
  if (e != cudaSuccess) return cuda_fail(e, "gb_apply_sinv");
  if (hst & gbk::kStTimeout) return fail(GB_ETIMEOUT, "a bounded wait for a staged factor tile gave up");
  return GB_OK;
}

}  // extern "C"

// ------------------------------------------------------------ true-residual check
// The recursive estimate ||rt_n|| / |pi^k_n| equals the true residual only
// while every inner solve is exact; an inexact S^-1 makes them drift apart.
// The check re-runs the listed columns in the same precision with the full
// history r_m kept on every row, forms x^k = sum_m c^k_m r_m for every shift
// (a complex GEMM of the history with the coefficients) and evaluates
// ||e_j - (z_k S - H) x^k||_2 in FP64 from the scalar CSR.
namespace {

// X[v][i][k] = sum_{m < nk[k]} c[m][k] r_m[i] for verified column v (panel
// v / C, slot v % C of W; r_m real: the real recurrence's v_m): 64 rows x 32 shifts per block, 16 history steps staged
// in shared memory per round, each thread 4 rows x 2 shifts.
template <bool REAL>
__global__ void __launch_bounds__(256) xk_kernel(int N4, int K, int C, int W, int Mcap, int nver, const char* team_ws,
                                                 size_t team_bytes, size_t o_hr, size_t o_cg, size_t o_nk,
                                                 const int* iters_max, double2* __restrict__ X) {
  using H = typename std::conditional<REAL, double, double2>::type;
  __shared__ H Rs[16][64];
  __shared__ double2 Cs[16][32];
  const int v = blockIdx.z, t = v / C, cc = v % C;
  const int i0 = blockIdx.x * 64, k0 = blockIdx.y * 32;
  const char* ws = team_ws + (size_t)t * team_bytes;
  const H* hr = reinterpret_cast<const H*>(ws + o_hr);
  const double2* cg = reinterpret_cast<const double2*>(ws + o_cg);
  const int* nk = reinterpret_cast<const int*>(ws + o_nk);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double2 acc[4][2];
  for (int a = 0; a < 4; ++a)
    for (int b = 0; b < 2; ++b) acc[a][b] = make_double2(0.0, 0.0);
  const int M = iters_max[v];
  for (int m0 = 0; m0 < M; m0 += 16) {
    for (int e = threadIdx.x; e < 16 * 64; e += 256) {
      const int mm = e >> 6, i = e & 63;
      const int m = m0 + mm, row = i0 + i;
      Rs[mm][i] = (m < M && row < N4) ? hr[(size_t)m * Mcap + (size_t)cc * N4 + row] : H{};
    }
    for (int e = threadIdx.x; e < 16 * 32; e += 256) {
      const int mm = e >> 5, kk = e & 31;
      const int m = m0 + mm, k = k0 + kk;
      Cs[mm][kk] = (k < K && m < nk[cc * K + k]) ? cg[((size_t)m * W + cc) * K + k] : make_double2(0.0, 0.0);
    }
    __syncthreads();
#pragma unroll 4
    for (int mm = 0; mm < 16; ++mm) {
      H r[4];
      double2 c[2];
      for (int a = 0; a < 4; ++a) r[a] = Rs[mm][ty * 4 + a];
      for (int b = 0; b < 2; ++b) c[b] = Cs[mm][tx * 2 + b];
      for (int a = 0; a < 4; ++a)
        for (int b = 0; b < 2; ++b) {
          if constexpr (REAL) {
            acc[a][b].x = fma(r[a], c[b].x, acc[a][b].x);
            acc[a][b].y = fma(r[a], c[b].y, acc[a][b].y);
          } else {
            acc[a][b].x = fma(r[a].x, c[b].x, fma(-r[a].y, c[b].y, acc[a][b].x));
            acc[a][b].y = fma(r[a].x, c[b].y, fma(r[a].y, c[b].x, acc[a][b].y));
          }
        }
    }
    __syncthreads();
  }
  for (int a = 0; a < 4; ++a)
    for (int b = 0; b < 2; ++b) {
      const int row = i0 + ty * 4 + a, k = k0 + tx * 2 + b;
      if (row < N4 && k < K) X[((size_t)v * N4 + row) * K + k] = acc[a][b];
    }
}

// res[k][v] = || e_j - (z_k S - H) x^k ||_2 from the scalar CSR, FP64; one
// block per (column, 32 shifts), lane = shift, warps split the rows, fixed
// reduction order.
__global__ void __launch_bounds__(256) true_resid_kernel(const gbk::DevMat mt, int N4, int K, int nver,
                                                         const int* __restrict__ cols, const double2* __restrict__ z,
                                                         const double2* __restrict__ X, double* __restrict__ res) {
  __shared__ double part[8][32];
  const int v = blockIdx.x, k = blockIdx.y * 32 + (threadIdx.x & 31), warp = threadIdx.x >> 5;
  const int j = cols[v];
  double acc = 0.0;
  if (k < K) {
    const double2 zk = z[k];
    const double2* Xv = X + (size_t)v * N4 * K;
    for (int i = warp; i < mt.n; i += 8) {
      double2 sx = make_double2(0.0, 0.0), hx = make_double2(0.0, 0.0);
      for (int t = mt.row_ptr[i]; t < mt.row_ptr[i + 1]; ++t) {
        const double2 xv = Xv[(size_t)mt.col_idx[t] * K + k];
        const double sv = mt.s_val[t], hv = mt.h_val[t];
        sx.x = fma(sv, xv.x, sx.x);
        sx.y = fma(sv, xv.y, sx.y);
        hx.x = fma(hv, xv.x, hx.x);
        hx.y = fma(hv, xv.y, hx.y);
      }
      // r_i = delta_ij - z_k (S x)_i + (H x)_i
      double rr = (i == j ? 1.0 : 0.0) - (zk.x * sx.x - zk.y * sx.y) + hx.x;
      double ri = -(zk.x * sx.y + zk.y * sx.x) + hx.y;
      acc = fma(rr, rr, fma(ri, ri, acc));
    }
  }
  part[warp][threadIdx.x & 31] = acc;
  __syncthreads();
  if (warp == 0 && k < K) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += part[w][threadIdx.x];
    res[(size_t)k * nver + v] = sqrt(s);
  }
}

struct VerLayout {
  Plan pl;
  int W;
  size_t o_x, o_im, o_cols, total;
};

gb_status ver_layout(const gb_matrix* m, const gb_solve_params* p, int32_t nver, VerLayout* L,
                     std::vector<int32_t>* cols_out, const int32_t* ver) {
  if (nver < 1 || nver > 1024) return fail(GB_EINVAL, "nver must be in [1, 1024]");
  gb_solve_params q = *p;
  std::vector<int32_t> cols(nver, 0);
  if (ver) {
    for (int i = 0; i < nver; ++i) {
      if (ver[i] < 0 || ver[i] >= p->nrhs) return fail(GB_EINVAL, "verify index %d out of range", i);
      cols[i] = p->rhs_cols[ver[i]];
    }
  } else {
    for (int i = 0; i < nver; ++i) cols[i] = p->rhs_cols[0];
  }
  int W = 1;
  while (W < 8 && W < nver) W <<= 1;
  q.nrhs = nver;
  q.rhs_cols = cols.data();
  q.panel = W;
  gb_status st = make_plan(m, &q, true, &L->pl, true, real_recurrence(m, p));
  if (st != GB_OK) return st;
  L->W = W;
  L->pl.teams = L->pl.npanels;  // verification: every panel at once, one team each
  size_t off = align256(L->pl.header_bytes) + L->pl.team_bytes * L->pl.teams;
  off = align256(off);
  L->o_x = off;
  off = align256(off + (size_t)nver * 4 * m->nb * p->nshift * 16);
  L->o_im = off;
  off = align256(off + sizeof(int) * nver);
  L->o_cols = off;
  off = align256(off + sizeof(int) * nver);
  L->total = off + 256;
  if (cols_out) *cols_out = cols;
  return GB_OK;
}

}  // namespace

extern "C" {

size_t gb_true_residual_workspace_size(const gb_matrix* m, const gb_solve_params* p, int32_t nver) {
  clear_error();
  if (!m || !p) {
    fail(GB_EINVAL, "NULL argument");
    return 0;
  }
  VerLayout L;
  if (ver_layout(m, p, nver, &L, nullptr, nullptr) != GB_OK) return 0;
  return L.total;
}

gb_status gb_true_residual(const gb_matrix* m, const gb_solve_params* p, int32_t nver, const int32_t* ver,
                           double* resid_true, const gb_outputs* out, void* workspace, size_t workspace_bytes,
                           void* stream, int32_t* nflagged) {
  clear_error();
  if (nflagged) *nflagged = 0;
  if (!m || !p || !ver || !resid_true) return fail(GB_EINVAL, "NULL argument");
  {
    Plan full;  // validates the parameters of the solve being checked
    const gb_status st = make_plan(m, p, false, &full);
    if (st != GB_OK) return st;
  }
  if (out && (!out->resid || !out->col_status))
    return fail(GB_EINVAL, "updating outputs needs their resid and col_status arrays");
  VerLayout L;
  std::vector<int32_t> cols;
  gb_status st = ver_layout(m, p, nver, &L, &cols, ver);
  if (st != GB_OK) return st;
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
    return fail(GB_EINVAL, "workspace must be a 256-byte aligned device pointer");
  if (workspace_bytes < L.total)
    return fail(GB_ENOMEM, "workspace too small: %zu < %zu bytes", workspace_bytes, L.total);
  int dev = 0;
  GB_CUDA(cudaGetDevice(&dev));
  if (dev != m->device) return fail(GB_EINVAL, "current device %d differs from the matrix's device %d", dev, m->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int K = p->nshift, N4 = 4 * (int)m->nb;
  const Plan& pl = L.pl;
  char* wsb = static_cast<char*>(workspace);
  // header: shifts (no weights), columns, offsets, status, counter
  std::vector<char> hdr(pl.header_bytes, 0);
  double2* hz = reinterpret_cast<double2*>(hdr.data() + pl.o_z);
  for (int k = 0; k < K; ++k) hz[k] = make_double2(p->z_re[k], p->z_im[k]);
  std::memcpy(hdr.data() + pl.o_cols, cols.data(), sizeof(int) * nver);
  long long* ho = reinterpret_cast<long long*>(hdr.data() + pl.o_off);
  ho[0] = 0;
  for (int i = 0; i < nver; ++i) ho[i + 1] = ho[i] + (m->h_row_ptr[cols[i] + 1] - m->h_row_ptr[cols[i]]);
  GB_CUDA(cudaMemcpyAsync(wsb, hdr.data(), pl.header_bytes, cudaMemcpyHostToDevice, s));
  GB_CUDA(cudaMemcpyAsync(wsb + L.o_cols, cols.data(), sizeof(int) * nver, cudaMemcpyHostToDevice, s));
  gbk::Args a = pl.a;
  a.m = m->dm;
  a.K = K;
  a.W = pl.W;
  a.KG = pl.KG;
  a.nrhs = nver;
  a.npanels = pl.npanels;
  a.maxit = p->maxit;
  a.inner_maxit = pl.inner_maxit;
  a.has_rho = 0;
  a.has_edm = 0;
  a.want_g = 1;
  a.full_hist = 1;
  a.tol = p->tol;
  a.itol = pl.itol;
  const int seed = p->seed_shift >= 0 ? p->seed_shift : K / 2;
  a.sigma = make_double2(p->z_re[seed], p->z_im[seed]);
  a.z = reinterpret_cast<const double2*>(wsb + pl.o_z);
  a.w_rho = reinterpret_cast<const double2*>(wsb + pl.o_wr);
  a.w_edm = reinterpret_cast<const double2*>(wsb + pl.o_we);
  a.rhs_cols = reinterpret_cast<const int*>(wsb + pl.o_cols);
  a.out_off = reinterpret_cast<const long long*>(wsb + pl.o_off);
  a.status = reinterpret_cast<int*>(wsb + pl.o_status);
  a.panel_counter = reinterpret_cast<int*>(wsb + pl.o_counter);
  a.team_ws = wsb + align256(pl.header_bytes);
  a.team_bytes = pl.team_bytes;
  a.Mcap = pl.Mcap;
  a.iters = reinterpret_cast<int*>(wsb + L.o_im);
  a.cg_smem = pl.cg_smem;
  if ((st = launch_team(a, p->prec == GB_FP64, pl.real, pl.teams, pl.threads, pl.dyn_smem, s)) != GB_OK) return st;
  double2* X = reinterpret_cast<double2*>(wsb + L.o_x);
  {
    const dim3 grid((unsigned)((N4 + 63) / 64), (unsigned)((K + 31) / 32), (unsigned)nver);
    if (pl.real)
      xk_kernel<true><<<grid, 256, 0, s>>>(N4, K, pl.C, 2 * pl.W, pl.Mcap, nver, a.team_ws, pl.team_bytes, a.o_hr,
                                           a.o_cg, a.o_nk, a.iters, X);
    else
      xk_kernel<false><<<grid, 256, 0, s>>>(N4, K, pl.C, pl.W, pl.Mcap, nver, a.team_ws, pl.team_bytes, a.o_hr, a.o_cg,
                                            a.o_nk, a.iters, X);
    GB_CUDA(cudaGetLastError());
  }
  {
    const dim3 grid((unsigned)nver, (unsigned)((K + 31) / 32));
    true_resid_kernel<<<grid, 256, 0, s>>>(m->dm, N4, K, nver, reinterpret_cast<const int*>(wsb + L.o_cols), a.z, X,
                                           resid_true);
    GB_CUDA(cudaGetLastError());
  }
  std::vector<int> vst(nver);
  GB_CUDA(cudaMemcpyAsync(vst.data(), a.status, sizeof(int) * nver, cudaMemcpyDeviceToHost, s));
  GB_CUDA(cudaStreamSynchronize(s));
  int any = 0;
  for (int v : vst) any |= v;
  if (any & gbk::kStTimeout) return fail(GB_ETIMEOUT, "a bounded wait for a staged factor tile gave up");
  if (out) {  // columns whose true residual misses tol become unconverged in `out`
    const int nrhs = p->nrhs;
    std::vector<double> rt((size_t)K * nver);
    GB_CUDA(cudaMemcpyAsync(rt.data(), resid_true, sizeof(double) * K * nver, cudaMemcpyDeviceToHost, s));
    std::vector<int32_t> cst(nrhs);
    GB_CUDA(cudaMemcpyAsync(cst.data(), out->col_status, sizeof(int32_t) * nrhs, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    int flagged = 0;
    for (int v = 0; v < nver; ++v) {
      const int c = ver[v];
      bool miss = false;
      for (int k = 0; k < K; ++k) miss |= !(rt[(size_t)k * nver + v] <= p->tol);
      if (!miss) continue;
      ++flagged;
      cst[c] |= gbk::kStNoConv;
      for (int k = 0; k < K; ++k) {
        const double r = rt[(size_t)k * nver + v];
        GB_CUDA(cudaMemcpyAsync(out->resid + (size_t)k * nrhs + c, &rt[(size_t)k * nver + v], sizeof(double),
                                cudaMemcpyHostToDevice, s));
        if (out->converged) {
          static const uint8_t zero = 0, one = 1;
          GB_CUDA(cudaMemcpyAsync(out->converged + (size_t)k * nrhs + c, r <= p->tol ? &one : &zero, 1,
                                  cudaMemcpyHostToDevice, s));
        }
      }
      GB_CUDA(cudaMemcpyAsync(out->col_status + c, &cst[c], sizeof(int32_t), cudaMemcpyHostToDevice, s));
    }
    GB_CUDA(cudaStreamSynchronize(s));
    if (nflagged) *nflagged = flagged;
  }
  return GB_OK;
}

}  // extern "C"

// ------------------------------------------------------------ chemical potential
// mu from the electron count and the Fermi-weighted rho / P^E of a finished
// solve of every orbital (Quantum molecular dynamics simulation: the density
// matrix of each MD step).  Real-axis rule on an evenly spaced shift grid
// z_k = eps_k + i eta, spacing d: c_k = -(s / pi) f((eps_k - mu) / kT) d,
// c^E_k = eps_k c_k, and N(mu) = sum_j q_j = -pi sum_k c_k D_k with the total
// DOS D_k = sum_j ldos[k][j], increasing in mu: bisection on the host over the
// K values D_k, then the reductions of rho / P^E / q / E on the device from
// the kept G_ij(z_k).
namespace {

__global__ void __launch_bounds__(256) dos_sum_kernel(const double* __restrict__ ldos, int K, int nrhs,
                                                      double* __restrict__ dos) {
  __shared__ double part[256];
  const int k = blockIdx.x;
  double acc = 0.0;
  for (int j = threadIdx.x; j < nrhs; j += 256) acc += ldos[(size_t)k * nrhs + j];
  part[threadIdx.x] = acc;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {  // fixed-order tree
    if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) dos[k] = part[0];
}

// rho_e = sum_k c_k Im G_e(z_k), edm_e = sum_k eps_k c_k Im G_e(z_k) for every
// kept pattern entry e (the weights are real).
__global__ void __launch_bounds__(256) fermi_density_kernel(const double2* __restrict__ g, long long P, int K,
                                                            const double* __restrict__ c,
                                                            const double* __restrict__ eps,
                                                            double* __restrict__ rho, double* __restrict__ edm) {
  const long long e = blockIdx.x * 256LL + threadIdx.x;
  if (e >= P) return;
  double r = 0.0, en = 0.0;
  for (int k = 0; k < K; ++k) {
    const double im = g[(size_t)k * P + e].y;
    r = fma(c[k], im, r);
    en = fma(eps[k] * c[k], im, en);
  }
  if (rho) rho[e] = r;
  if (edm) edm[e] = en;
}

__global__ void __launch_bounds__(256) local_sums_kernel(const gbk::DevMat m, const int* __restrict__ cols,
                                                         const long long* __restrict__ off, int nrhs,
                                                         const double* __restrict__ rho, double* __restrict__ q,
                                                         double* __restrict__ el) {
  const int c = blockIdx.x * 256 + threadIdx.x;
  if (c >= nrhs) return;
  const int j = cols[c], base = m.row_ptr[j], mc = m.row_ptr[j + 1] - base;
  double qs = 0.0, es = 0.0;
  for (int t = 0; t < mc; ++t) {
    const double r = rho[off[c] + t];
    qs = fma(r, m.s_val[base + t], qs);
    es = fma(r, m.h_val[base + t], es);
  }
  if (q) q[c] = qs;
  if (el) el[c] = es;
}

double fermi_f(double x) { return x >= 0 ? std::exp(-x) / (1.0 + std::exp(-x)) : 1.0 / (1.0 + std::exp(x)); }

}  // namespace

extern "C" {

size_t gb_fermi_workspace_size(const gb_matrix* m, const gb_solve_params* p) {
  clear_error();
  if (!m || !p || p->nshift < 1 || p->nrhs < 1) {
    fail(GB_EINVAL, "NULL argument or empty problem");
    return 0;
  }
  return align256(8 * (size_t)p->nshift) * 3 + align256(4 * (size_t)p->nrhs) + align256(8 * ((size_t)p->nrhs + 1)) +
         256;
}

gb_status gb_fermi_density(const gb_matrix* m, const gb_solve_params* p, const double* g_proj, const double* ldos,
                           double n_electrons, double kT, double spin, double* mu, const gb_outputs* out,
                           void* workspace, size_t workspace_bytes, void* stream) {
  clear_error();
  if (!m || !p || !g_proj || !ldos || !mu || !out) return fail(GB_EINVAL, "NULL argument");
  if (misaligned(g_proj, 16) || misaligned(ldos, 8) || check_outputs(out) != GB_OK)
    return fail(GB_EINVAL, "g_proj must be 16-byte aligned and every other array to its element");
  const int K = p->nshift, nrhs = p->nrhs;
  if (K < 2 || !p->z_re || !p->z_im) return fail(GB_EINVAL, "need at least two shifts");
  if (nrhs != m->n || !p->rhs_cols) return fail(GB_EINVAL, "the electron count needs every orbital solved (nrhs = n)");
  {
    std::vector<char> seen(m->n, 0);
    for (int c = 0; c < nrhs; ++c) {
      const int j = p->rhs_cols[c];
      if (j < 0 || j >= m->n || seen[j]) return fail(GB_EINVAL, "rhs_cols must hold every orbital once");
      seen[j] = 1;
    }
  }
  const double d = (p->z_re[K - 1] - p->z_re[0]) / (K - 1);
  if (!(d > 0.0)) return fail(GB_EINVAL, "shift real parts must increase");
  for (int k = 0; k < K; ++k)
    if (!std::isfinite(p->z_re[k]) || std::fabs(p->z_re[k] - (p->z_re[0] + k * d)) > 1e-9 * std::fabs(d) * K ||
        !(p->z_im[k] > 0.0))
      return fail(GB_EINVAL, "the shifts must be evenly spaced in Re z with Im z > 0");
  if (!(kT > 0.0) || !(spin > 0.0) || !(n_electrons > 0.0) || !(n_electrons < spin * m->n))
    return fail(GB_EINVAL, "need kT > 0, spin > 0 and 0 < n_electrons < spin * n");
  const size_t need = gb_fermi_workspace_size(m, p);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
    return fail(GB_EINVAL, "workspace must be a 256-byte aligned device pointer");
  if (workspace_bytes < need) return fail(GB_ENOMEM, "workspace too small: %zu < %zu bytes", workspace_bytes, need);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(workspace);
  double* d_dos = reinterpret_cast<double*>(w);
  double* d_c = reinterpret_cast<double*>(w + align256(8 * (size_t)K));
  double* d_eps = reinterpret_cast<double*>(w + 2 * align256(8 * (size_t)K));
  int* d_cols = reinterpret_cast<int*>(w + 3 * align256(8 * (size_t)K));
  long long* d_off = reinterpret_cast<long long*>(w + 3 * align256(8 * (size_t)K) + align256(4 * (size_t)nrhs));
  dos_sum_kernel<<<K, 256, 0, s>>>(ldos, K, nrhs, d_dos);
  GB_CUDA(cudaGetLastError());
  std::vector<double> dos(K);
  GB_CUDA(cudaMemcpyAsync(dos.data(), d_dos, sizeof(double) * K, cudaMemcpyDeviceToHost, s));
  GB_CUDA(cudaStreamSynchronize(s));
  auto count = [&](double x) {
    double n = 0.0;
    for (int k = 0; k < K; ++k) n += spin * fermi_f((p->z_re[k] - x) / kT) * d * dos[k];  // -pi c_k D_k
    return n;
  };
  double lo = p->z_re[0] - 40.0 * kT, hi = p->z_re[K - 1] + 40.0 * kT;
  if (!(count(lo) <= n_electrons && n_electrons <= count(hi)))
    return fail(GB_EINVAL, "the electron count is outside what the shift grid can hold (%g..%g)", count(lo), count(hi));
  for (int it = 0; it < 200; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (count(mid) < n_electrons)
      lo = mid;
    else
      hi = mid;
  }
  *mu = 0.5 * (lo + hi);
  std::vector<double> c(K), eps(K);
  for (int k = 0; k < K; ++k) {
    eps[k] = p->z_re[k];
    c[k] = -(spin / 3.141592653589793238462643383279502884) * fermi_f((eps[k] - *mu) / kT) * d;
  }
  std::vector<long long> off(nrhs + 1, 0);
  for (int i = 0; i < nrhs; ++i) {
    const int j = p->rhs_cols[i];
    off[i + 1] = off[i] + (m->h_row_ptr[j + 1] - m->h_row_ptr[j]);
  }
  const long long P = off[nrhs];
  GB_CUDA(cudaMemcpyAsync(d_c, c.data(), sizeof(double) * K, cudaMemcpyHostToDevice, s));
  GB_CUDA(cudaMemcpyAsync(d_eps, eps.data(), sizeof(double) * K, cudaMemcpyHostToDevice, s));
  GB_CUDA(cudaMemcpyAsync(d_cols, p->rhs_cols, sizeof(int) * nrhs, cudaMemcpyHostToDevice, s));
  GB_CUDA(cudaMemcpyAsync(d_off, off.data(), sizeof(long long) * (nrhs + 1), cudaMemcpyHostToDevice, s));
  fermi_density_kernel<<<(unsigned)((P + 255) / 256), 256, 0, s>>>(reinterpret_cast<const double2*>(g_proj), P, K,
                                                                   d_c, d_eps, out->rho, out->edm);
  GB_CUDA(cudaGetLastError());
  if (out->rho && (out->q || out->e_loc)) {
    local_sums_kernel<<<(unsigned)((nrhs + 255) / 256), 256, 0, s>>>(m->dm, d_cols, d_off, nrhs, out->rho, out->q,
                                                                     out->e_loc);
    GB_CUDA(cudaGetLastError());
  }
  GB_CUDA(cudaStreamSynchronize(s));  // the host vectors above are this call's locals
  return GB_OK;
}

}  // extern "C"

// ------------------------------------------------------------ correction solve
// Shifted COCG with one seed can stagnate for a shift whose shifted residual
// loses attainable accuracy (observed near the gap of some PPV-like chains at
// eta = 0.02).  The correction re-solves each such column alone in plain FP64
// (exact factor inner solve) with its worst unconverged shift as the seed, so
// that shift's residual is the seed's own.  If shifts still miss tol, it
// repeats with the worst remaining shift as the next seed (up to six seeds)
// and keeps, per shift, the result of the seed that served it best; the
// column's outputs are then formed from those G_ij(z_k).
namespace {

struct CorrLayout {
  size_t plan_total, o_ldos, o_rho, o_edm, o_q, o_e, o_it, o_conv, o_res, o_g, o_in, o_st, total;
};

// Workspace of one single-column FP64 correction solve (its plan depends on
// maxit, the shift count and the longest pattern row, not on the column)
// followed by that column's temporary outputs.
gb_status corr_layout(const gb_matrix* m, const gb_solve_params* p, bool want_g, CorrLayout* L) {
  if (!p->rhs_cols || p->nrhs < 1) return fail(GB_EINVAL, "rhs_cols must hold nrhs >= 1 columns");
  gb_solve_params q = *p;
  const int32_t col0 = p->rhs_cols[0];
  q.nrhs = 1;
  q.rhs_cols = &col0;
  q.prec = GB_FP64;
  q.seed_shift = -1;
  q.panel = 1;
  q.flags = 0;
  q.inner_tol = 0.0;
  Plan pl;
  (void)want_g;
  const gb_status st = make_plan(m, &q, true, &pl);
  if (st != GB_OK) return st;
  const size_t K = p->nshift, mr = (size_t)std::max(m->max_row, 1);
  size_t off = align256(pl.total);
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = align256(off + bytes);
    return o;
  };
  L->plan_total = pl.total;
  L->o_ldos = take(K * 8);
  L->o_rho = take(mr * 8);
  L->o_edm = take(mr * 8);
  L->o_q = take(8);
  L->o_e = take(8);
  L->o_it = take(4);
  L->o_conv = take(K);
  L->o_res = take(K * 8);
  L->o_g = take(K * mr * 16);  // always: the per-shift merge over seeds needs G on the pattern row
  L->o_in = take(4);
  L->o_st = take(4);
  L->total = off + 256;
  return GB_OK;
}

}  // namespace

extern "C" {

size_t gb_correct_workspace_size(const gb_matrix* m, const gb_solve_params* p, int32_t want_g) {
  clear_error();
  if (!m || !p) {
    fail(GB_EINVAL, "NULL argument");
    return 0;
  }
  CorrLayout L;
  if (corr_layout(m, p, want_g != 0, &L) != GB_OK) return 0;
  return L.total;
}

gb_status gb_correct_unconverged(const gb_matrix* m, const gb_solve_params* p, const gb_outputs* out,
                                 void* workspace, size_t workspace_bytes, void* stream, int32_t* ncorrected) {
  clear_error();
  if (ncorrected) *ncorrected = 0;
  if (!m || !p || !out) return fail(GB_EINVAL, "NULL argument");
  if (!out->col_status || !out->resid) return fail(GB_EINVAL, "col_status and resid of the first solve are required");
  {
    Plan full;  // validates every parameter of the first solve
    const gb_status st = make_plan(m, p, out->g_proj != nullptr, &full);
    if (st != GB_OK) return st;
  }
  const bool want_g = out->g_proj != nullptr;
  CorrLayout L;
  gb_status st = corr_layout(m, p, want_g, &L);
  if (st != GB_OK) return st;
  if (!workspace) return fail(GB_EINVAL, "workspace is NULL");
  if ((reinterpret_cast<uintptr_t>(workspace) & 255) != 0) return fail(GB_EINVAL, "workspace must be 256-byte aligned");
  if (workspace_bytes < L.total)
    return fail(GB_ENOMEM, "workspace too small: %zu < %zu bytes", workspace_bytes, L.total);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int K = p->nshift, nrhs = p->nrhs;
  std::vector<int32_t> hst(nrhs);
  std::vector<double> hres((size_t)K * nrhs);
  std::vector<uint8_t> hconv(out->converged ? (size_t)K * nrhs : 0);
  GB_CUDA(cudaMemcpyAsync(hst.data(), out->col_status, sizeof(int32_t) * nrhs, cudaMemcpyDeviceToHost, s));
  GB_CUDA(cudaMemcpyAsync(hres.data(), out->resid, sizeof(double) * K * nrhs, cudaMemcpyDeviceToHost, s));
  if (out->converged)
    GB_CUDA(cudaMemcpyAsync(hconv.data(), out->converged, (size_t)K * nrhs, cudaMemcpyDeviceToHost, s));
  GB_CUDA(cudaStreamSynchronize(s));
  const std::vector<int64_t>& rp = m->h_row_ptr;
  std::vector<long long> off(nrhs + 1, 0);
  for (int c = 0; c < nrhs; ++c) {
    const int j = p->rhs_cols[c];
    off[c + 1] = off[c] + (rp[j + 1] - rp[j]);
  }
  const long long P = off[nrhs];
  char* wsb = static_cast<char*>(workspace);
  int fixed = 0, left = 0;
  constexpr int kMaxSeeds = 6;
  for (int c = 0; c < nrhs; ++c) {
    const int sc = hst[c];
    if (!(sc & gbk::kStNoConv) || (sc & (gbk::kStBreakdown | gbk::kStNotSPD))) continue;
    const int32_t col = p->rhs_cols[c];
    const long long mc = off[c + 1] - off[c];
    // per shift, the best FP64 result over the seeds tried so far
    std::vector<double> best(K, INFINITY), tres(K);
    std::vector<double2> bestg((size_t)K * mc), tg((size_t)K * mc);
    std::vector<double> cur(K);  // residuals that pick the next seed
    for (int k = 0; k < K; ++k) {
      const size_t e = (size_t)k * nrhs + c;
      const bool conv = out->converged ? hconv[e] != 0 : hres[e] <= p->tol;
      cur[k] = conv ? 0.0 : hres[e];
    }
    int it_sum = 0, in_sum = 0, rounds = 0;
    bool done = false;
    std::vector<char> tried(K, 0);
    for (int round = 0; round < kMaxSeeds && !done; ++round) {
      // First the first solve's own seed, now in FP64 with the exact inner
      // solve (this alone converges most stalled columns); then the worst
      // shift still missing tol that has not been a seed yet.  (A shift that
      // stalls as a non-seed shift can stall as the seed too, so the worst
      // shift is not the first choice.)
      int kw = -1;
      if (round == 0) {
        kw = p->seed_shift >= 0 ? p->seed_shift : K / 2;
      } else {
        double rw = -1.0;
        for (int k = 0; k < K; ++k)
          if (!tried[k] && cur[k] > p->tol && cur[k] > rw) {
            rw = cur[k];
            kw = k;
          }
        if (kw < 0) break;  // every failing shift has been a seed
      }
      tried[kw] = 1;
      gb_solve_params q = *p;
      q.nrhs = 1;
      q.rhs_cols = &col;
      q.prec = GB_FP64;
      q.seed_shift = kw;
      q.panel = 1;
      q.flags = kFlagStall;  // a stalled column stops early and tries the next seed
      q.inner_tol = 0.0;
      gb_outputs t{};
      t.ldos = out->ldos ? reinterpret_cast<double*>(wsb + L.o_ldos) : nullptr;
      t.rho = out->rho ? reinterpret_cast<double*>(wsb + L.o_rho) : nullptr;
      t.edm = out->edm ? reinterpret_cast<double*>(wsb + L.o_edm) : nullptr;
      t.q = out->q ? reinterpret_cast<double*>(wsb + L.o_q) : nullptr;
      t.e_loc = out->e_loc ? reinterpret_cast<double*>(wsb + L.o_e) : nullptr;
      t.iters = reinterpret_cast<int32_t*>(wsb + L.o_it);
      t.converged = out->converged ? reinterpret_cast<uint8_t*>(wsb + L.o_conv) : nullptr;
      t.resid = reinterpret_cast<double*>(wsb + L.o_res);
      t.g_proj = reinterpret_cast<double*>(wsb + L.o_g);
      t.inner_iters = reinterpret_cast<int32_t*>(wsb + L.o_in);
      t.col_status = reinterpret_cast<int32_t*>(wsb + L.o_st);
      const gb_status sub = gb_shifted_solve(m, &q, &t, workspace, L.plan_total, stream);
      if (sub != GB_OK && sub != GB_ENOCONV) return sub;
      int hit = 0, hin = 0;
      GB_CUDA(cudaMemcpyAsync(tres.data(), t.resid, sizeof(double) * K, cudaMemcpyDeviceToHost, s));
      GB_CUDA(cudaMemcpyAsync(tg.data(), t.g_proj, sizeof(double2) * K * mc, cudaMemcpyDeviceToHost, s));
      GB_CUDA(cudaMemcpyAsync(&hit, t.iters, sizeof(int), cudaMemcpyDeviceToHost, s));
      GB_CUDA(cudaMemcpyAsync(&hin, t.inner_iters, sizeof(int), cudaMemcpyDeviceToHost, s));
      GB_CUDA(cudaStreamSynchronize(s));
      it_sum += hit;
      in_sum += hin;
      ++rounds;
      if (round == 0 && sub == GB_OK) {
        // one seed converged every shift: the solve's own outputs are the column's
        auto column = [&](void* dst, const void* src, size_t esz) {  // [K][nrhs] column c <- [K][1]
          return cudaMemcpy2DAsync(static_cast<char*>(dst) + esz * c, esz * nrhs, src, esz, esz, K,
                                   cudaMemcpyDeviceToDevice, s);
        };
        auto one = [&](void* dst, const void* src, size_t esz) {
          return cudaMemcpyAsync(static_cast<char*>(dst) + esz * c, src, esz, cudaMemcpyDeviceToDevice, s);
        };
        if (out->ldos) GB_CUDA(column(out->ldos, t.ldos, sizeof(double)));
        if (out->converged) GB_CUDA(column(out->converged, t.converged, 1));
        GB_CUDA(column(out->resid, t.resid, sizeof(double)));
        if (out->rho) GB_CUDA(cudaMemcpyAsync(out->rho + off[c], t.rho, sizeof(double) * mc, cudaMemcpyDeviceToDevice, s));
        if (out->edm) GB_CUDA(cudaMemcpyAsync(out->edm + off[c], t.edm, sizeof(double) * mc, cudaMemcpyDeviceToDevice, s));
        if (out->q) GB_CUDA(one(out->q, t.q, sizeof(double)));
        if (out->e_loc) GB_CUDA(one(out->e_loc, t.e_loc, sizeof(double)));
        if (out->iters) GB_CUDA(one(out->iters, t.iters, sizeof(int32_t)));
        if (out->inner_iters) GB_CUDA(one(out->inner_iters, t.inner_iters, sizeof(int32_t)));
        GB_CUDA(one(out->col_status, t.col_status, sizeof(int32_t)));
        if (want_g)
          GB_CUDA(cudaMemcpy2DAsync(out->g_proj + 2 * off[c], 16 * (size_t)P, t.g_proj, 16 * (size_t)mc,
                                    16 * (size_t)mc, K, cudaMemcpyDeviceToDevice, s));
        // the next column's solve reuses the temporaries: stream-ordered after these copies
        GB_CUDA(cudaStreamSynchronize(s));
        done = true;
        break;
      }
      bool all = true;
      for (int k = 0; k < K; ++k) {
        if (tres[k] < best[k]) {
          best[k] = tres[k];
          for (long long t2 = 0; t2 < mc; ++t2) bestg[(size_t)k * mc + t2] = tg[(size_t)k * mc + t2];
        }
        cur[k] = best[k];
        all &= best[k] <= p->tol;
      }
      if (all) done = true;
    }
    if (rounds > 1 || !done) {
      // Several seeds: every shift keeps the result of the seed that served it
      // best, and the column's outputs are formed from those G_ij(z_k) on the
      // pattern row (the same reductions as the solve's final phase).
      std::vector<double> sv(mc), hv(mc);
      const int base = (int)rp[col];
      GB_CUDA(cudaMemcpyAsync(sv.data(), m->dm.s_val + base, sizeof(double) * mc, cudaMemcpyDeviceToHost, s));
      GB_CUDA(cudaMemcpyAsync(hv.data(), m->dm.h_val + base, sizeof(double) * mc, cudaMemcpyDeviceToHost, s));
      GB_CUDA(cudaStreamSynchronize(s));
      std::vector<double> ldos(K), rho(mc, 0.0), edm(mc, 0.0);
      std::vector<uint8_t> conv(K);
      for (int k = 0; k < K; ++k) {
        double im = 0.0;
        for (long long t2 = 0; t2 < mc; ++t2) im += bestg[(size_t)k * mc + t2].y * sv[t2];
        ldos[k] = -im / 3.141592653589793238462643383279502884;
        conv[k] = best[k] <= p->tol ? 1 : 0;
        const double wr_re = p->w_rho ? p->w_rho[2 * k] : 0.0, wr_im = p->w_rho ? p->w_rho[2 * k + 1] : 0.0;
        const double we_re = p->w_edm ? p->w_edm[2 * k] : 0.0, we_im = p->w_edm ? p->w_edm[2 * k + 1] : 0.0;
        for (long long t2 = 0; t2 < mc; ++t2) {
          const double2 g = bestg[(size_t)k * mc + t2];
          rho[t2] += wr_re * g.y + wr_im * g.x;  // Im(c g)
          edm[t2] += we_re * g.y + we_im * g.x;
        }
      }
      double qs = 0.0, es = 0.0;
      for (long long t2 = 0; t2 < mc; ++t2) {
        qs += rho[t2] * sv[t2];
        es += rho[t2] * hv[t2];
      }
      const bool allc = std::all_of(conv.begin(), conv.end(), [](uint8_t v) { return v != 0; });
      const int32_t cst = allc ? 0 : gbk::kStNoConv;
      done = allc;
      for (int k = 0; k < K; ++k) {
        const size_t e = (size_t)k * nrhs + c;
        if (out->ldos) GB_CUDA(cudaMemcpyAsync(out->ldos + e, &ldos[k], sizeof(double), cudaMemcpyHostToDevice, s));
        if (out->converged) GB_CUDA(cudaMemcpyAsync(out->converged + e, &conv[k], 1, cudaMemcpyHostToDevice, s));
        GB_CUDA(cudaMemcpyAsync(out->resid + e, &best[k], sizeof(double), cudaMemcpyHostToDevice, s));
        if (want_g)
          GB_CUDA(cudaMemcpyAsync(out->g_proj + 2 * ((size_t)k * P + off[c]), &bestg[(size_t)k * mc],
                                  sizeof(double2) * mc, cudaMemcpyHostToDevice, s));
      }
      if (out->rho && p->w_rho)
        GB_CUDA(cudaMemcpyAsync(out->rho + off[c], rho.data(), sizeof(double) * mc, cudaMemcpyHostToDevice, s));
      if (out->edm && p->w_edm)
        GB_CUDA(cudaMemcpyAsync(out->edm + off[c], edm.data(), sizeof(double) * mc, cudaMemcpyHostToDevice, s));
      if (out->q && p->w_rho) GB_CUDA(cudaMemcpyAsync(out->q + c, &qs, sizeof(double), cudaMemcpyHostToDevice, s));
      if (out->e_loc && p->w_rho) GB_CUDA(cudaMemcpyAsync(out->e_loc + c, &es, sizeof(double), cudaMemcpyHostToDevice, s));
      if (out->iters) GB_CUDA(cudaMemcpyAsync(out->iters + c, &it_sum, sizeof(int32_t), cudaMemcpyHostToDevice, s));
      if (out->inner_iters)
        GB_CUDA(cudaMemcpyAsync(out->inner_iters + c, &in_sum, sizeof(int32_t), cudaMemcpyHostToDevice, s));
      GB_CUDA(cudaMemcpyAsync(out->col_status + c, &cst, sizeof(int32_t), cudaMemcpyHostToDevice, s));
      GB_CUDA(cudaStreamSynchronize(s));  // the host buffers above are this iteration's locals
    }
    if (done)
      ++fixed;
    else
      ++left;
  }
  GB_CUDA(cudaStreamSynchronize(s));
  if (ncorrected) *ncorrected = fixed;
  if (left > 0)
    return fail(GB_ENOCONV, "%d column(s) still miss tol after the FP64 correction solve", left);
  return GB_OK;
}

}  // extern "C"

// ------------------------------------------------------------ allocation-free solve
// gb_shifted_solve_static: the same solve for callers that may not allocate
// memory once they are running — e.g. an application whose device memory is
// owned by another runtime's pool that claims the whole GPU, or a latency-
// critical loop in which cudaMalloc's implicit device synchronisation is not
// acceptable.  Its device scratch is one file-scope array below; its host-side
// staging uses fixed static buffers.  Nothing here calls cudaMalloc, cudaFree
// or any other allocating routine.
#include <mutex>

namespace {

constexpr size_t kStaticScratchBytes = size_t(32) << 20;  // 32 MiB per device
constexpr int kStaticMaxRhs = 4096;
constexpr int kMaxDevices = 64;

// Device scratch shared by every gb_shifted_solve_static call on a device.  In
// host code this name is only a stand-in for the symbol: its device address is
// obtained once per device with cudaGetSymbolAddress below.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

std::mutex g_static_mu;                      // guards the table and the host staging buffers
void* g_static_addr[kMaxDevices] = {nullptr};  // device address of g_static_scratch per device
alignas(256) char g_static_hdr[256 * 1024];  // host staging of the launch header
int g_static_status[kStaticMaxRhs];          // host copy of the per-column status

}  // namespace

extern "C" {

gb_status gb_shifted_solve_static(const gb_matrix* m, const gb_solve_params* p, const gb_outputs* out,
                                  void* stream) {
  clear_error();
  if (!out) return fail(GB_EINVAL, "outputs is NULL");
  if (!p) return fail(GB_EINVAL, "params is NULL");
  if (check_outputs(out) != GB_OK) return GB_EINVAL;
  if (p->nrhs > kStaticMaxRhs) return fail(GB_EINVAL, "nrhs %d exceeds the static limit %d", p->nrhs, kStaticMaxRhs);
  Plan pl;
  const bool want_g = out->g_proj != nullptr;
  gb_status st = make_plan(m, p, want_g, &pl);
  if (st != GB_OK) return st;
  // The library's choice of panels for the real recurrence is made for time: room for two
  // columns at least, and more up to one wave, and a team's records (16 K (maxit + 1) bytes a
  // column with g_proj) grow with them.  Where they do not fit, the seed recurrence's choice of
  // width, which starts at one column, may.
  if (p->panel <= 0 && pl.real && align256(pl.header_bytes) + pl.team_bytes > kStaticScratchBytes) {
    Plan alt;
    if ((st = make_plan(m, p, want_g, &alt, false, 0)) != GB_OK) return st;
    gb_solve_params narrow = *p;
    narrow.panel = alt.C;
    if ((st = make_plan(m, &narrow, want_g, &alt)) != GB_OK) return st;
    if (alt.team_bytes < pl.team_bytes) pl = alt;
  }
  int dev = 0;
  GB_CUDA(cudaGetDevice(&dev));
  if (dev != m->device) return fail(GB_EINVAL, "current device %d differs from the matrix's device %d", dev, m->device);
  if (dev < 0 || dev >= kMaxDevices) return fail(GB_EINVAL, "device ordinal %d out of range", dev);
  if (pl.header_bytes > sizeof(g_static_hdr)) return fail(GB_EINVAL, "too many shifts/columns for the static path");
  // fewer teams than the allocating path if needed: results do not depend on it
  const size_t hdr_al = align256(pl.header_bytes);
  if (hdr_al + pl.team_bytes > kStaticScratchBytes)
    return fail(GB_ENOMEM, "problem needs %zu bytes of scratch per team; the static scratch holds %zu bytes",
                hdr_al + pl.team_bytes, kStaticScratchBytes);
  const int teams = (int)std::min<size_t>(pl.teams, (kStaticScratchBytes - hdr_al) / pl.team_bytes);

  std::lock_guard<std::mutex> lock(g_static_mu);
  if (g_static_addr[dev] == nullptr) {  // first call on this device: look up the scratch address
    void* ptr = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_scratch);
    if (e != cudaSuccess || ptr == nullptr) return cuda_fail(e, "cudaGetSymbolAddress(static scratch)");
    g_static_addr[dev] = ptr;
  }
  char* wsb = static_cast<char*>(g_static_addr[dev]);
  cudaStream_t s = static_cast<cudaStream_t>(stream);

  const int K = p->nshift, nrhs = p->nrhs;
  std::memset(g_static_hdr, 0, pl.header_bytes);  // includes the panel counter, which must start at 0
  double2* hz = reinterpret_cast<double2*>(g_static_hdr + pl.o_z);
  double2* hwr = reinterpret_cast<double2*>(g_static_hdr + pl.o_wr);
  double2* hwe = reinterpret_cast<double2*>(g_static_hdr + pl.o_we);
  for (int k = 0; k < K; ++k) {
    hz[k] = make_double2(p->z_re[k], p->z_im[k]);
    hwr[k] = p->w_rho ? make_double2(p->w_rho[2 * k], p->w_rho[2 * k + 1]) : make_double2(0, 0);
    hwe[k] = p->w_edm ? make_double2(p->w_edm[2 * k], p->w_edm[2 * k + 1]) : make_double2(0, 0);
  }
  std::memcpy(g_static_hdr + pl.o_cols, p->rhs_cols, sizeof(int) * nrhs);
  long long* ho = reinterpret_cast<long long*>(g_static_hdr + pl.o_off);
  ho[0] = 0;
  for (int i = 0; i < nrhs; ++i) {
    const int j = p->rhs_cols[i];
    ho[i + 1] = ho[i] + (m->h_row_ptr[j + 1] - m->h_row_ptr[j]);
  }
  GB_CUDA(cudaMemcpyAsync(wsb, g_static_hdr, pl.header_bytes, cudaMemcpyHostToDevice, s));

  gbk::Args& a = pl.a;
  a.m = m->dm;
  a.K = K;
  a.W = pl.W;
  a.KG = pl.KG;
  a.nrhs = nrhs;
  a.npanels = pl.npanels;
  a.maxit = p->maxit;
  a.inner_maxit = pl.inner_maxit;
  a.has_rho = p->w_rho != nullptr;
  a.has_edm = p->w_edm != nullptr;
  a.want_g = want_g;
  a.tol = p->tol;
  a.itol = pl.itol;
  const int seed = p->seed_shift >= 0 ? p->seed_shift : K / 2;
  a.sigma = make_double2(p->z_re[seed], p->z_im[seed]);
  a.z = reinterpret_cast<const double2*>(wsb + pl.o_z);
  a.w_rho = reinterpret_cast<const double2*>(wsb + pl.o_wr);
  a.w_edm = reinterpret_cast<const double2*>(wsb + pl.o_we);
  a.rhs_cols = reinterpret_cast<const int*>(wsb + pl.o_cols);
  a.out_off = reinterpret_cast<const long long*>(wsb + pl.o_off);
  a.status = reinterpret_cast<int*>(wsb + pl.o_status);
  a.panel_counter = reinterpret_cast<int*>(wsb + pl.o_counter);
  a.team_ws = wsb + hdr_al;
  a.team_bytes = pl.team_bytes;
  a.Mcap = pl.Mcap;
  a.ldos = out->ldos;
  a.rho = out->rho;
  a.edm = out->edm;
  a.q = out->q;
  a.e_loc = out->e_loc;
  a.iters = out->iters;
  a.inner_iters = out->inner_iters;
  a.col_status = out->col_status;
  a.conv = out->converged;
  a.resid = out->resid;
  a.g_proj = reinterpret_cast<double2*>(out->g_proj);
  a.P = ho[nrhs];
  a.cg_smem = pl.cg_smem;
  if ((st = launch_team(a, p->prec == GB_FP64, pl.real, teams, pl.threads, pl.dyn_smem, s)) != GB_OK) return st;
  GB_CUDA(cudaMemcpyAsync(g_static_status, a.status, sizeof(int) * nrhs, cudaMemcpyDeviceToHost, s));
  GB_CUDA(cudaStreamSynchronize(s));
  int any = 0;
  for (int i = 0; i < nrhs; ++i) any |= g_static_status[i];
  if (any & gbk::kStTimeout) return fail(GB_ETIMEOUT, "a bounded wait for a staged factor tile gave up");
  if (any & gbk::kStNotSPD) return fail(GB_ENOTSPD, "inner CG found S not positive definite");
  if (any & gbk::kStBreakdown) return fail(GB_EBREAKDOWN, "COCG breakdown in at least one column");
  if (any & (gbk::kStNoConv | gbk::kStInner))
    return fail(GB_ENOCONV, "some (shift, column) pairs did not reach tol within maxit%s",
                (any & gbk::kStInner) ? " (inner CG hit its cap)" : "");
  return GB_OK;
}

size_t gb_static_scratch_bytes(void) { return kStaticScratchBytes; }

}  // extern "C"

// ------------------------------------------------------------ batched solve
// Many independent systems in one persistent launch (team_kernel_batched).
namespace {

struct BatchPlan {
  int C, W, teams, threads, total_panels, maxK, maxit, Mcap, KG;
  bool real, mixed, want_g;
  size_t N4, team_bytes, header_bytes, total, dyn_smem;
  std::vector<int> order;  // systems, largest estimated cost first
  gbk::Args proto;
};

// A system's estimated time in a batch: its iterations grow like n^0.6 (152 to 912
// orbitals: 396 to 1130) and the time of each like n, beside the shift polynomials.
double batch_cost(const gb_matrix* m, const gb_solve_params* p) {
  const double n = (double)m->n;
  return std::pow(n, 0.6) * (n + 0.25 * p->nshift);
}

// The panel width of a mixed batch on wide teams, one per SM, at most C.  A batch of
// unequal systems waits for its largest, whose panels get faster with fewer columns (24
// systems: 290, 220, 181 ms with 8, 4, 2), while the small ones can share SMs: so a
// narrower width is taken where the modelled finishing time of the work queue (largest
// first) is at least 12 % shorter.  GB300, uneven chains of 8 columns, 8 / 4 / 2 columns a
// panel: 96 of up to 32 monomers 446 / 354 / 379 ms (taken: 4), 40 398 / 308 / 265 (2), 60
// of up to 20 240 / 189 / 151 (2), 150 of up to 12 161 / 137 / 234 (4).
int batch_width(int nsys, const gb_matrix* const* mats, const gb_solve_params* params, const std::vector<int>& order,
                int nsm, int C) {
  auto relative = [](int cols) { return cols == 8 ? 1.6 : cols == 4 ? 1.21 : cols == 2 ? 1.0 : 0.3 * cols; };
  double best = 0.0;
  int width = C;
  for (int cand = C; cand >= 2; cand /= 2) {
    std::vector<double> busy((size_t)nsm, 0.0);  // a heap, the first SM to be free on top
    long long panels = 0;
    for (int s = 0; s < nsys; ++s) panels += (params[s].nrhs + cand - 1) / cand;
    if (panels > 8LL * nsm) break;
    double end = 0.0;
    for (int q = 0; q < nsys; ++q) {
      const int s = order[q];
      const double t = relative(cand) * batch_cost(mats[s], &params[s]);
      for (int k = (params[s].nrhs + cand - 1) / cand; k > 0; --k) {
        std::pop_heap(busy.begin(), busy.end(), std::greater<double>());
        busy.back() += t;
        end = std::max(end, busy.back());
        std::push_heap(busy.begin(), busy.end(), std::greater<double>());
      }
    }
    if (best > 0.0 && end >= 0.88 * best) continue;
    best = end;
    width = cand;
  }
  return width;
}

gb_status make_batch_plan(int32_t nsys, const gb_matrix* const* mats, const gb_solve_params* params,
                          const gb_outputs* outs, int32_t panel, BatchPlan* bp) {
  if (nsys < 1 || !mats || !params) return fail(GB_EINVAL, "need nsys >= 1, mats and params");
  const gb_precision prec = params[0].prec;
  size_t n4max = 0;
  int kmax = 0, itmax = 0, rowmax = 0, dev = -1;
  long long cols = 0;
  bool want_g = false;
  for (int s = 0; s < nsys; ++s) {
    Plan pl;
    gb_status st = make_plan(mats[s], &params[s], false, &pl);
    if (st != GB_OK) {
      char msg[sizeof(gb::g_err)];
      std::snprintf(msg, sizeof msg, "%s", gb::g_err);
      return fail(st, "system %d: %s", s, msg);
    }
    if (params[s].prec != prec) return fail(GB_EINVAL, "all systems must use the same precision");
    if (dev >= 0 && mats[s]->device != dev) return fail(GB_EINVAL, "all matrices must live on one device");
    dev = mats[s]->device;
    n4max = std::max(n4max, 4 * (size_t)mats[s]->nb);
    kmax = std::max(kmax, (int)params[s].nshift);
    itmax = std::max(itmax, (int)params[s].maxit);
    rowmax = std::max(rowmax, (int)mats[s]->max_row);
    cols += params[s].nrhs;
    if (outs && outs[s].g_proj) want_g = true;
  }
  cudaDeviceProp prop;
  cudaError_t e = cudaGetDeviceProperties(&prop, dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDeviceProperties");
  const int nsm = prop.multiProcessorCount;
  bool real = true;  // one recurrence per launch (batch_parts)
  for (int s = 0; s < nsys; ++s) real = real && real_recurrence(mats[s], &params[s]);
  auto width = [&](int cols) { return real ? std::max(1, cols / 2) : cols; };
  const void* fn = batched_fn(prec == GB_FP64, real);
  // dynamic shared memory: the factor solve's buffers (systems without a
  // factor leave them unused)
  auto dyn_bytes = [&](int w) -> size_t { return gbk::dyn_layout(prec == GB_FP64, w, true, 0, 63, !real).bytes; };
  auto occupancy = [&](size_t dyn) {
    int per_sm = 1;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, gbk::TPB, dyn) != cudaSuccess || per_sm < 1)
      per_sm = 1;
    return per_sm;
  };
  // largest systems first for load balance
  bp->order.resize(nsys);
  for (int s = 0; s < nsys; ++s) bp->order[s] = s;
  std::stable_sort(bp->order.begin(), bp->order.end(),
                   [&](int x, int y) { return batch_cost(mats[x], &params[x]) > batch_cost(mats[y], &params[y]); });
  int C = panel;
  bool wide = false;  // wide teams, one per SM
  if (C <= 0) {  // widest panel that still gives every resident team a work item
    auto panels = [&](int cand) {
      long long np = 0;
      for (int s = 0; s < nsys; ++s) np += (params[s].nrhs + cand - 1) / cand;
      return np;
    };
    int cap = 2;  // wider panels would stay partly empty in every system
    for (int s = 0; s < nsys; ++s)
      while (cap < 32 && cap < params[s].nrhs) cap *= 2;
    C = 1;
    if (real && prec == GB_MIXED) {
      // wide teams where one wave holds every panel (as in make_plan), or where no system
      // has more than 8 columns: 300 chains of 8, wide teams / 512 threads, 8 columns a
      // panel 303 / 367 ms, 4 columns 382 / 322
      C = 2;
      while (C < cap && panels(C) > nsm) C *= 2;
      wide = panels(C) <= nsm || C == 8;
      if (wide) C = batch_width(nsys, mats, params, bp->order, nsm, C);
    }
    if (!wide) {
      C = 1;
      for (int cand : {32, 16, 8, 4, 2})
        if (cand <= cap && 4 * panels(cand) >= 3LL * nsm * occupancy(dyn_bytes(width(cand)))) {
          C = cand;
          break;
        }
    }
    if (real && C == 1) C = 2;  // a pair costs what one of its columns does
  }
  if (C != 1 && C != 2 && C != 4 && C != 8 && C != 16 && C != 32)
    return fail(GB_EINVAL, "panel must be 1, 2, 4, 8, 16 or 32");
  const int W = width(C);
  bp->dyn_smem = dyn_bytes(W);
  const int per_sm = occupancy(bp->dyn_smem);
  bp->C = C;
  bp->real = real;
  bp->W = W;
  bp->mixed = prec == GB_MIXED;
  bp->want_g = want_g;
  bp->N4 = n4max;
  bp->maxK = kmax;
  bp->KG = (kmax + 31) / 32;
  bp->maxit = itmax;
  bp->Mcap = C * rowmax;
  std::memset(&bp->proto, 0, sizeof bp->proto);
  bp->team_bytes = layout_team(n4max, W, kmax, bp->KG, itmax, bp->Mcap, want_g, real, bp->proto);
  bp->proto.C = C;
  bp->total_panels = 0;
  for (int s = 0; s < nsys; ++s) bp->total_panels += (params[s].nrhs + C - 1) / C;
  wide = wide || (real && prec != GB_FP64 && bp->total_panels <= nsm);
  bp->teams = std::min(bp->total_panels, wide ? nsm : nsm * per_sm);
  bp->threads = wide ? gbk::TPB_WIDE : gbk::TPB;
  // header: descriptors, panel prefix, counter, then per-system arrays
  size_t hb = align256(sizeof(gbk::Args) * nsys) + align256(sizeof(int) * (nsys + 1)) + 256;
  for (int s = 0; s < nsys; ++s)
    hb += 3 * align256(16 * (size_t)params[s].nshift) + align256(sizeof(int) * params[s].nrhs) +
          align256(sizeof(long long) * (params[s].nrhs + 1)) + align256(sizeof(int) * params[s].nrhs);
  bp->header_bytes = hb;
  bp->total = hb + bp->team_bytes * bp->teams + 256;
  return GB_OK;
}

// The systems of a batch that one launch solves.  A system's own parameters say by which
// recurrence it is solved, alone, in any batch and when gb_true_residual runs it again; a
// batch that holds both kinds takes two launches, one after the other in the same workspace.
struct BatchPart {
  BatchPlan plan;
  std::vector<const gb_matrix*> mats;
  std::vector<gb_solve_params> params;
  std::vector<gb_outputs> outs;  // empty: a size query without g_proj
};
gb_status batch_parts(int32_t nsys, const gb_matrix* const* mats, const gb_solve_params* params,
                      const gb_outputs* outs, int32_t panel, std::vector<BatchPart>* parts) {
  BatchPlan whole;  // checks every argument, in the caller's numbering
  gb_status st = make_batch_plan(nsys, mats, params, outs, panel, &whole);
  if (st != GB_OK) return st;
  for (const bool real : {true, false}) {
    BatchPart part;
    for (int s = 0; s < nsys; ++s) {
      if (real_recurrence(mats[s], &params[s]) != real) continue;
      part.mats.push_back(mats[s]);
      part.params.push_back(params[s]);
      if (outs) part.outs.push_back(outs[s]);
    }
    const int32_t n = (int32_t)part.mats.size();
    if (n == 0) continue;
    if (n == nsys)
      part.plan = whole;
    else if ((st = make_batch_plan(n, part.mats.data(), part.params.data(), outs ? part.outs.data() : nullptr, panel,
                                   &part.plan)) != GB_OK)
      return st;
    parts->push_back(std::move(part));
  }
  return GB_OK;
}
size_t parts_total(const std::vector<BatchPart>& parts) {
  size_t total = 0;
  for (const BatchPart& p : parts) total = std::max(total, p.plan.total);
  return total;
}

// One part's launch; its columns' status bits are added to *any.  Synchronous.
gb_status run_part(const BatchPart& part, char* wsb, cudaStream_t s, int* any) {
  const BatchPlan& bp = part.plan;
  int nsys = (int)part.mats.size();
  const gb_matrix* const* mats = part.mats.data();
  const gb_solve_params* params = part.params.data();
  const gb_outputs* outs = part.outs.data();
  std::vector<char> hdr(bp.header_bytes, 0);
  gbk::Args* desc = reinterpret_cast<gbk::Args*>(hdr.data());
  size_t off = align256(sizeof(gbk::Args) * nsys);
  int* prefix = reinterpret_cast<int*>(hdr.data() + off);
  const size_t o_prefix = off;
  off += align256(sizeof(int) * (nsys + 1));
  const size_t o_counter = off;
  off += 256;
  std::vector<size_t> o_status(nsys);
  prefix[0] = 0;
  char* team_ws = wsb + align256(bp.header_bytes);
  for (int q = 0; q < nsys; ++q) {
    const int sidx = bp.order[q];
    const gb_matrix* m = mats[sidx];
    const gb_solve_params* p = &params[sidx];
    const gb_outputs* out = &outs[sidx];
    const int K = p->nshift, nrhs = p->nrhs;
    const size_t o_z = off;
    off += align256(16 * (size_t)K);
    const size_t o_wr = off;
    off += align256(16 * (size_t)K);
    const size_t o_we = off;
    off += align256(16 * (size_t)K);
    const size_t o_cols = off;
    off += align256(sizeof(int) * nrhs);
    const size_t o_off = off;
    off += align256(sizeof(long long) * (nrhs + 1));
    o_status[sidx] = off;
    off += align256(sizeof(int) * nrhs);
    double2* hz = reinterpret_cast<double2*>(hdr.data() + o_z);
    double2* hwr = reinterpret_cast<double2*>(hdr.data() + o_wr);
    double2* hwe = reinterpret_cast<double2*>(hdr.data() + o_we);
    for (int k = 0; k < K; ++k) {
      hz[k] = make_double2(p->z_re[k], p->z_im[k]);
      hwr[k] = p->w_rho ? make_double2(p->w_rho[2 * k], p->w_rho[2 * k + 1]) : make_double2(0, 0);
      hwe[k] = p->w_edm ? make_double2(p->w_edm[2 * k], p->w_edm[2 * k + 1]) : make_double2(0, 0);
    }
    std::memcpy(hdr.data() + o_cols, p->rhs_cols, sizeof(int) * nrhs);
    long long* ho = reinterpret_cast<long long*>(hdr.data() + o_off);
    ho[0] = 0;
    for (int i = 0; i < nrhs; ++i) {
      const int j = p->rhs_cols[i];
      ho[i + 1] = ho[i] + (m->h_row_ptr[j + 1] - m->h_row_ptr[j]);
    }
    gbk::Args a = bp.proto;  // workspace regions laid out for the maxima
    {
      gbk::Args im;
      set_inner_method(m, p, p->inner_tol > 0 ? p->inner_tol : (p->prec == GB_FP64 ? 1e-14 : 1e-7), bp.real, im);
      a.inner_cheb = im.inner_cheb;
      a.inner_dense = im.inner_dense;
      a.inner_bchol = im.inner_bchol;
      a.bc_levels = im.bc_levels;
      a.hp_fp32 = im.hp_fp32;
      a.stall = im.stall;
      a.bc_bw_alloc = 63;  // the launch's shared memory is sized for any band
      a.cheb_K = im.cheb_K;
      a.cheb_c0 = im.cheb_c0;
      std::memcpy(a.cheb_A, im.cheb_A, sizeof a.cheb_A);
      std::memcpy(a.cheb_B, im.cheb_B, sizeof a.cheb_B);
    }
    a.m = m->dm;
    a.K = K;
    a.W = bp.W;
    a.KG = (K + 31) / 32;
    a.nrhs = nrhs;
    a.npanels = (nrhs + bp.C - 1) / bp.C;
    a.maxit = p->maxit;
    a.inner_maxit = 500;
    a.has_rho = p->w_rho != nullptr;
    a.has_edm = p->w_edm != nullptr;
    a.want_g = out->g_proj != nullptr;
    a.tol = p->tol;
    a.itol = p->inner_tol > 0 ? p->inner_tol : (p->prec == GB_FP64 ? 1e-14 : 1e-7);
    const int seed = p->seed_shift >= 0 ? p->seed_shift : K / 2;
    a.sigma = make_double2(p->z_re[seed], p->z_im[seed]);
    a.z = reinterpret_cast<const double2*>(wsb + o_z);
    a.w_rho = reinterpret_cast<const double2*>(wsb + o_wr);
    a.w_edm = reinterpret_cast<const double2*>(wsb + o_we);
    a.rhs_cols = reinterpret_cast<const int*>(wsb + o_cols);
    a.out_off = reinterpret_cast<const long long*>(wsb + o_off);
    a.status = reinterpret_cast<int*>(wsb + o_status[sidx]);
    a.panel_counter = reinterpret_cast<int*>(wsb + o_counter);
    a.team_ws = team_ws;
    a.team_bytes = bp.team_bytes;
    a.Mcap = bp.C * m->max_row;
    a.cg_smem = 0;
    a.ldos = out->ldos;
    a.rho = out->rho;
    a.edm = out->edm;
    a.q = out->q;
    a.e_loc = out->e_loc;
    a.iters = out->iters;
    a.inner_iters = out->inner_iters;
    a.col_status = out->col_status;
    a.conv = out->converged;
    a.resid = out->resid;
    a.g_proj = reinterpret_cast<double2*>(out->g_proj);
    a.P = ho[nrhs];
    desc[q] = a;
    prefix[q + 1] = prefix[q] + a.npanels;
  }
  GB_CUDA(cudaMemcpyAsync(wsb, hdr.data(), bp.header_bytes, cudaMemcpyHostToDevice, s));
  const gbk::Args* d_desc = reinterpret_cast<const gbk::Args*>(wsb);
  const int* d_prefix = reinterpret_cast<const int*>(wsb + o_prefix);
  int* d_counter = reinterpret_cast<int*>(wsb + o_counter);
  {
    const void* fn = batched_fn(!bp.mixed, bp.real);
    GB_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bp.dyn_smem));
    size_t team_bytes = bp.team_bytes;
    void* args[] = {&d_desc, &d_prefix, &nsys, &d_counter, &team_ws, &team_bytes};
    GB_CUDA(cudaLaunchKernel(fn, dim3(bp.teams), dim3(bp.threads), args, bp.dyn_smem, s));
  }
  GB_CUDA(cudaMemcpyAsync(hdr.data(), wsb, bp.header_bytes, cudaMemcpyDeviceToHost, s));
  GB_CUDA(cudaStreamSynchronize(s));
  for (int q = 0; q < nsys; ++q) {
    const int* hs = reinterpret_cast<const int*>(hdr.data() + o_status[q]);
    for (int i = 0; i < params[q].nrhs; ++i) *any |= hs[i];
  }
  return GB_OK;
}

}  // namespace

extern "C" {

size_t gb_batched_workspace_size(int32_t nsys, const gb_matrix* const* mats, const gb_solve_params* params,
                                 int32_t panel, int32_t want_g) {
  clear_error();
  std::vector<BatchPart> parts;
  std::vector<gb_outputs> fake;
  if (want_g && nsys > 0) {
    fake.assign(nsys, gb_outputs{});
    for (auto& f : fake) f.g_proj = reinterpret_cast<double*>(1);
  }
  if (batch_parts(nsys, mats, params, want_g ? fake.data() : nullptr, panel, &parts) != GB_OK) return 0;
  return parts_total(parts);
}

gb_status gb_shifted_solve_batched(int32_t nsys, const gb_matrix* const* mats, const gb_solve_params* params,
                                   const gb_outputs* outs, int32_t panel, void* workspace, size_t workspace_bytes,
                                   void* stream) {
  clear_error();
  if (!outs) return fail(GB_EINVAL, "outputs is NULL");
  for (int i = 0; i < nsys; ++i)
    if (check_outputs(&outs[i]) != GB_OK) return GB_EINVAL;
  std::vector<BatchPart> parts;
  gb_status st = batch_parts(nsys, mats, params, outs, panel, &parts);
  if (st != GB_OK) return st;
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
    return fail(GB_EINVAL, "workspace must be a 256-byte aligned device pointer");
  const size_t need = parts_total(parts);
  if (workspace_bytes < need) return fail(GB_ENOMEM, "workspace too small: %zu < %zu bytes", workspace_bytes, need);
  int dev = 0;
  GB_CUDA(cudaGetDevice(&dev));
  if (dev != mats[0]->device) return fail(GB_EINVAL, "current device differs from the matrices' device");
  int any = 0;
  for (const BatchPart& part : parts)
    if ((st = run_part(part, static_cast<char*>(workspace), static_cast<cudaStream_t>(stream), &any)) != GB_OK) return st;
  if (any & gbk::kStTimeout) return fail(GB_ETIMEOUT, "a bounded wait for a staged factor tile gave up");
  if (any & gbk::kStNotSPD) return fail(GB_ENOTSPD, "inner CG found S not positive definite");
  if (any & gbk::kStBreakdown) return fail(GB_EBREAKDOWN, "COCG breakdown in at least one column");
  if (any & (gbk::kStNoConv | gbk::kStInner))
    return fail(GB_ENOCONV, "some (shift, column) pairs did not reach tol within maxit%s",
                (any & gbk::kStInner) ? " (inner CG hit its cap)" : "");
  return GB_OK;
}

gb_status gb_tune_panel_batched(int32_t nsys, const gb_matrix* const* mats, const gb_solve_params* params,
                                const gb_outputs* outs, int32_t probe_maxit, void* workspace,
                                size_t workspace_bytes, void* stream, int32_t* best_panel, float* times_ms) {
  clear_error();
  if (!best_panel || nsys < 1 || probe_maxit < 1) return fail(GB_EINVAL, "bad tuner arguments");
  std::vector<gb_solve_params> probe(params, params + nsys);
  for (auto& p : probe) p.maxit = std::min(p.maxit, probe_maxit);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaEvent_t e0, e1;
  GB_CUDA(cudaEventCreate(&e0));
  GB_CUDA(cudaEventCreate(&e1));
  // the configuration's panel widths {8, 16, 32, 64} less 64: a 64-column
  // panel's per-column shared state next to the factor solve's buffers would
  // leave one team per SM instead of two
  const int cands[3] = {8, 16, 32};
  float best = 1e30f;
  *best_panel = 0;
  for (int i = 0; i < 3; ++i) {
    if (times_ms) times_ms[i] = -1.f;
    std::vector<BatchPart> parts;
    if (batch_parts(nsys, mats, probe.data(), outs, cands[i], &parts) != GB_OK || parts_total(parts) > workspace_bytes)
      continue;
    cudaEventRecord(e0, s);
    const gb_status st = gb_shifted_solve_batched(nsys, mats, probe.data(), outs, cands[i], workspace,
                                                  workspace_bytes, stream);
    cudaEventRecord(e1, s);
    cudaEventSynchronize(e1);
    if (st != GB_OK && st != GB_ENOCONV) continue;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (times_ms) times_ms[i] = ms;
    if (ms < best) {
      best = ms;
      *best_panel = cands[i];
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  clear_error();
  if (*best_panel == 0) return fail(GB_ENOMEM, "no candidate panel width fits the workspace");
  return GB_OK;
}

}  // extern "C"

// ------------------------------------------------------------ batched correction
// The correction of a finished batched launch: every column that missed tol,
// of every system, is solved again in one batched FP64 launch (exact inner
// solve, the first solve's seed, one column per panel), and the columns that
// now meet tol are copied into the batch's outputs.  Columns that still miss
// tol then go through gb_correct_unconverged (seed switching), system by
// system.  The layout of the temporaries depends on which columns failed, so
// the plan reads every system's col_status first.
namespace {

struct CorrBatch {
  std::vector<int> sys;                      // sub-system -> system
  std::vector<std::vector<int32_t>> cols;    // failing orbital columns per sub-system
  std::vector<std::vector<int>> cidx;        // their positions in the system's column list
  std::vector<std::vector<long long>> soff;  // packed pattern offsets of the sub-system
  std::vector<gb_solve_params> q;
  std::vector<gb_outputs> t;                 // temporaries, as offsets from the workspace base
  size_t tmp_bytes = 0, batch_bytes = 0, single_bytes = 0, total = 0;
};

gb_status corr_batch_plan(int32_t nsys, const gb_matrix* const* mats, const gb_solve_params* params,
                          const gb_outputs* outs, cudaStream_t s, CorrBatch* cb) {
  if (nsys < 1 || !mats || !params || !outs) return fail(GB_EINVAL, "NULL argument or empty batch");
  for (int i = 0; i < nsys; ++i) {
    const gb_solve_params* p = &params[i];
    if (!mats[i] || !outs[i].col_status || !outs[i].resid || !p->rhs_cols || p->nrhs < 1)
      return fail(GB_EINVAL, "system %d: matrix, col_status, resid and rhs_cols are required", i);
    std::vector<int32_t> st(p->nrhs);
    GB_CUDA(cudaMemcpyAsync(st.data(), outs[i].col_status, sizeof(int32_t) * p->nrhs, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    std::vector<int32_t> fc;
    std::vector<int> ci;
    for (int c = 0; c < p->nrhs; ++c)
      if ((st[c] & gbk::kStNoConv) && !(st[c] & (gbk::kStBreakdown | gbk::kStNotSPD))) {
        fc.push_back(p->rhs_cols[c]);
        ci.push_back(c);
      }
    if (fc.empty()) continue;
    cb->sys.push_back(i);
    cb->cols.push_back(std::move(fc));
    cb->cidx.push_back(std::move(ci));
  }
  const int nsub = (int)cb->sys.size();
  size_t off = 0;
  cb->q.resize(nsub);
  cb->t.assign(nsub, gb_outputs{});
  cb->soff.resize(nsub);
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += align256(bytes);
    return reinterpret_cast<void*>(o + 256);  // +256: a null offset stays distinguishable
  };
  for (int u = 0; u < nsub; ++u) {
    const int i = cb->sys[u];
    const gb_matrix* m = mats[i];
    const gb_outputs& o = outs[i];
    gb_solve_params q = params[i];
    q.nrhs = (int32_t)cb->cols[u].size();
    q.rhs_cols = cb->cols[u].data();
    q.prec = GB_FP64;
    q.panel = 1;
    q.flags = kFlagStall;  // a stalled column stops early and tries the next seed
    q.inner_tol = 0.0;
    cb->q[u] = q;
    const size_t K = q.nshift, n = q.nrhs;
    std::vector<long long>& so = cb->soff[u];
    so.assign(n + 1, 0);
    for (size_t c = 0; c < n; ++c) {
      const int j = cb->cols[u][c];
      so[c + 1] = so[c] + (m->h_row_ptr[j + 1] - m->h_row_ptr[j]);
    }
    const size_t P = so[n];
    gb_outputs& t = cb->t[u];
    if (o.ldos) t.ldos = static_cast<double*>(take(8 * K * n));
    if (o.rho) t.rho = static_cast<double*>(take(8 * P));
    if (o.edm) t.edm = static_cast<double*>(take(8 * P));
    if (o.q) t.q = static_cast<double*>(take(8 * n));
    if (o.e_loc) t.e_loc = static_cast<double*>(take(8 * n));
    t.iters = static_cast<int32_t*>(take(4 * n));
    t.inner_iters = static_cast<int32_t*>(take(4 * n));
    t.col_status = static_cast<int32_t*>(take(4 * n));
    if (o.converged) t.converged = static_cast<uint8_t*>(take(K * n));
    t.resid = static_cast<double*>(take(8 * K * n));
    if (o.g_proj) t.g_proj = static_cast<double*>(take(16 * K * P));
  }
  cb->tmp_bytes = align256(off + 256);
  bool want_g = false;
  for (int u = 0; u < nsub; ++u) want_g |= outs[cb->sys[u]].g_proj != nullptr;
  if (nsub > 0) {
    std::vector<const gb_matrix*> sm(nsub);
    for (int u = 0; u < nsub; ++u) sm[u] = mats[cb->sys[u]];
    cb->batch_bytes = gb_batched_workspace_size(nsub, sm.data(), cb->q.data(), 1, want_g ? 1 : 0);
    if (cb->batch_bytes == 0) return GB_EINVAL;  // error text set by the size call
    for (int u = 0; u < nsub; ++u) {
      const int i = cb->sys[u];
      const size_t b = gb_correct_workspace_size(mats[i], &params[i], outs[i].g_proj != nullptr);
      if (b == 0) return GB_EINVAL;
      cb->single_bytes = std::max(cb->single_bytes, b);
    }
  }
  cb->total = std::max(cb->tmp_bytes + cb->batch_bytes, cb->single_bytes);
  return GB_OK;
}

template <typename T>
T* at(void* base, T* rel) {
  return rel ? reinterpret_cast<T*>(static_cast<char*>(base) + (reinterpret_cast<uintptr_t>(rel) - 256)) : nullptr;
}

}  // namespace

extern "C" {

size_t gb_correct_batched_workspace_size(int32_t nsys, const gb_matrix* const* mats, const gb_solve_params* params,
                                         const gb_outputs* outs, void* stream) {
  clear_error();
  CorrBatch cb;
  if (corr_batch_plan(nsys, mats, params, outs, static_cast<cudaStream_t>(stream), &cb) != GB_OK) return 0;
  return std::max<size_t>(cb.total, 256);
}

gb_status gb_correct_batched(int32_t nsys, const gb_matrix* const* mats, const gb_solve_params* params,
                             const gb_outputs* outs, void* workspace, size_t workspace_bytes, void* stream,
                             int32_t* ncorrected) {
  clear_error();
  if (ncorrected) *ncorrected = 0;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  CorrBatch cb;
  gb_status st = corr_batch_plan(nsys, mats, params, outs, s, &cb);
  if (st != GB_OK) return st;
  const int nsub = (int)cb.sys.size();
  if (nsub == 0) return GB_OK;
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
    return fail(GB_EINVAL, "workspace must be a 256-byte aligned device pointer");
  if (workspace_bytes < cb.total) return fail(GB_ENOMEM, "workspace too small: %zu < %zu bytes", workspace_bytes, cb.total);
  char* base = static_cast<char*>(workspace);
  std::vector<gb_outputs> tv(nsub);
  std::vector<const gb_matrix*> sm(nsub);
  for (int u = 0; u < nsub; ++u) {
    const gb_outputs& r = cb.t[u];
    gb_outputs& t = tv[u];
    t.ldos = at(base, r.ldos);
    t.rho = at(base, r.rho);
    t.edm = at(base, r.edm);
    t.q = at(base, r.q);
    t.e_loc = at(base, r.e_loc);
    t.iters = at(base, r.iters);
    t.inner_iters = at(base, r.inner_iters);
    t.col_status = at(base, r.col_status);
    t.converged = at(base, r.converged);
    t.resid = at(base, r.resid);
    t.g_proj = at(base, r.g_proj);
    sm[u] = mats[cb.sys[u]];
  }
  st = gb_shifted_solve_batched(nsub, sm.data(), cb.q.data(), tv.data(), 1, base + cb.tmp_bytes, cb.batch_bytes,
                                stream);
  if (st != GB_OK && st != GB_ENOCONV) return st;
  int fixed = 0;
  std::vector<int> left;
  for (int u = 0; u < nsub; ++u) {
    const int i = cb.sys[u];
    const gb_solve_params* p = &params[i];
    const gb_outputs& o = outs[i];
    const gb_outputs& t = tv[u];
    const int n = cb.q[u].nrhs, K = p->nshift, nrhs = p->nrhs;
    std::vector<int32_t> tst(n);
    GB_CUDA(cudaMemcpyAsync(tst.data(), t.col_status, sizeof(int32_t) * n, cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    // packed offsets of the system's own column list
    std::vector<long long> ooff(nrhs + 1, 0);
    for (int c = 0; c < nrhs; ++c) {
      const int j = p->rhs_cols[c];
      ooff[c + 1] = ooff[c] + (mats[i]->h_row_ptr[j + 1] - mats[i]->h_row_ptr[j]);
    }
    const long long Po = ooff[nrhs], Pt = cb.soff[u][n];
    bool rest = false;
    for (int a = 0; a < n; ++a) {
      if (tst[a] & (gbk::kStNoConv | gbk::kStBreakdown | gbk::kStNotSPD)) {
        rest = true;
        continue;
      }
      const int c = cb.cidx[u][a];
      const long long mc = ooff[c + 1] - ooff[c];
      auto col2d = [&](void* dst, const void* src, size_t esz) {  // [K][nrhs] column c <- [K][n] column a
        return cudaMemcpy2DAsync(static_cast<char*>(dst) + esz * c, esz * nrhs,
                                 static_cast<const char*>(src) + esz * a, esz * n, esz, K, cudaMemcpyDeviceToDevice, s);
      };
      auto one = [&](void* dst, const void* src, size_t esz) {
        return cudaMemcpyAsync(static_cast<char*>(dst) + esz * c, static_cast<const char*>(src) + esz * a, esz,
                               cudaMemcpyDeviceToDevice, s);
      };
      if (o.ldos) GB_CUDA(col2d(o.ldos, t.ldos, 8));
      if (o.converged) GB_CUDA(col2d(o.converged, t.converged, 1));
      GB_CUDA(col2d(o.resid, t.resid, 8));
      if (o.rho)
        GB_CUDA(cudaMemcpyAsync(o.rho + ooff[c], t.rho + cb.soff[u][a], 8 * mc, cudaMemcpyDeviceToDevice, s));
      if (o.edm)
        GB_CUDA(cudaMemcpyAsync(o.edm + ooff[c], t.edm + cb.soff[u][a], 8 * mc, cudaMemcpyDeviceToDevice, s));
      if (o.q) GB_CUDA(one(o.q, t.q, 8));
      if (o.e_loc) GB_CUDA(one(o.e_loc, t.e_loc, 8));
      if (o.iters) GB_CUDA(one(o.iters, t.iters, 4));
      if (o.inner_iters) GB_CUDA(one(o.inner_iters, t.inner_iters, 4));
      GB_CUDA(one(o.col_status, t.col_status, 4));
      if (o.g_proj)
        GB_CUDA(cudaMemcpy2DAsync(o.g_proj + 2 * ooff[c], 16 * (size_t)Po, t.g_proj + 2 * cb.soff[u][a],
                                  16 * (size_t)Pt, 16 * (size_t)mc, K, cudaMemcpyDeviceToDevice, s));
      ++fixed;
    }
    if (rest) left.push_back(i);
  }
  GB_CUDA(cudaStreamSynchronize(s));  // the temporaries are reused below
  bool all = true;
  for (const int i : left) {
    int32_t f = 0;
    const gb_status r = gb_correct_unconverged(mats[i], &params[i], &outs[i], workspace, workspace_bytes, stream, &f);
    fixed += f;
    if (r == GB_ENOCONV) {
      all = false;
    } else if (r != GB_OK) {
      if (ncorrected) *ncorrected = fixed;
      return r;
    }
  }
  if (ncorrected) *ncorrected = fixed;
  if (!all) return fail(GB_ENOCONV, "some columns still miss tol after the FP64 correction solves");
  return GB_OK;
}

}  // extern "C"

// ------------------------------------------------------------ atomic forces
// F_a = -Tr[rho dH/dR_a] + Tr[P^E dS/dR_a] (Quantum molecular dynamics
// simulation: the forces of each MD step) from the rho / P^E of a solve of
// every orbital.  For two-center elements the gradient of entry (j, i) with
// respect to the atom of row j is grad[:, e] (e its CSR position) and with
// respect to the atom of i its negative; the element (i, j) is the same
// function, so the trace over both orders gives
//   F_a = -sum_{j in a} sum_{i in R_j, atom(i) != a} ((rho_ij + rho_ji) gH_e - (P^E_ij + P^E_ji) gS_e),
// rho_ij read from column j of the packed output and rho_ji from column i (the
// two differ by the solve's rounding; the sum keeps the trace exact for the
// matrix as computed).  One warp per atom; the lanes take the entries of its
// orbitals' pattern rows and reduce in a fixed order (deterministic).
namespace {

__global__ void __launch_bounds__(256) forces_kernel(const gbk::DevMat m, const int* __restrict__ atom_off,
                                                     const int* __restrict__ orb_atom, const int* __restrict__ col_of,
                                                     const long long* __restrict__ off,
                                                     const long long* __restrict__ tpos, const double* __restrict__ rho,
                                                     const double* __restrict__ edm, const double* __restrict__ gh,
                                                     const double* __restrict__ gs, long long nnz, int n_atoms,
                                                     double* __restrict__ F) {
  const int a = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  if (a >= n_atoms) return;  // uniform per warp
  const int lane = threadIdx.x & 31;
  double fx = 0.0, fy = 0.0, fz = 0.0;
  for (int j = atom_off[a]; j < atom_off[a + 1]; ++j) {
    const int c = col_of[j], e0 = m.row_ptr[j], e1 = m.row_ptr[j + 1];
    const long long base = off[c] - e0;  // packed index of entry e in column j: base + e
    for (int e = e0 + lane; e < e1; e += 32) {
      if (orb_atom[m.col_idx[e]] == a) continue;
      const long long o = tpos[e];  // the same element in column i
      const double r = rho[base + e] + rho[o], q = edm[base + e] + edm[o];
      fx = fma(q, gs[e], fma(-r, gh[e], fx));
      fy = fma(q, gs[nnz + e], fma(-r, gh[nnz + e], fy));
      fz = fma(q, gs[2 * nnz + e], fma(-r, gh[2 * nnz + e], fz));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    fx += __shfl_xor_sync(0xffffffffu, fx, o);
    fy += __shfl_xor_sync(0xffffffffu, fy, o);
    fz += __shfl_xor_sync(0xffffffffu, fz, o);
  }
  if (lane == 0) {
    F[3 * a] = fx;
    F[3 * a + 1] = fy;
    F[3 * a + 2] = fz;
  }
}

}  // namespace

extern "C" {

size_t gb_forces_workspace_size(const gb_matrix* m, const gb_solve_params* p, int32_t n_atoms) {
  clear_error();
  if (!m || !p || p->nrhs < 1 || n_atoms < 1) {
    fail(GB_EINVAL, "NULL argument, no columns or no atoms");
    return 0;
  }
  return align256(4 * ((size_t)n_atoms + 1)) + 2 * align256(4 * (size_t)m->n) +
         align256(8 * ((size_t)p->nrhs + 1)) + align256(8 * (size_t)m->nnz) + 256;
}

gb_status gb_forces(const gb_matrix* m, const gb_solve_params* p, const double* rho, const double* edm,
                    const double* grad_h, const double* grad_s, const int64_t* atom_off, int32_t n_atoms,
                    double* forces, void* workspace, size_t workspace_bytes, void* stream) {
  clear_error();
  if (!m || !p || !rho || !edm || !grad_h || !grad_s || !atom_off || !forces) return fail(GB_EINVAL, "NULL argument");
  if (misaligned(rho, 8) || misaligned(edm, 8) || misaligned(grad_h, 8) || misaligned(grad_s, 8) ||
      misaligned(forces, 8))
    return fail(GB_EINVAL, "arrays must be aligned to their element");
  const int n = (int)m->n, nrhs = p->nrhs;
  if (n_atoms < 1 || atom_off[0] != 0 || atom_off[n_atoms] != n)
    return fail(GB_EINVAL, "atom_off must run from 0 to n over n_atoms atoms");
  for (int a = 0; a < n_atoms; ++a)
    if (atom_off[a + 1] <= atom_off[a]) return fail(GB_EINVAL, "atom %d has no orbitals", a);
  if (nrhs != n || !p->rhs_cols) return fail(GB_EINVAL, "forces need every orbital solved (nrhs = n)");
  std::vector<int> col_of(n, -1), orb_atom(n), aoff(n_atoms + 1);
  for (int c = 0; c < nrhs; ++c) {
    const int j = p->rhs_cols[c];
    if (j < 0 || j >= n || col_of[j] >= 0) return fail(GB_EINVAL, "rhs_cols must hold every orbital once");
    col_of[j] = c;
  }
  for (int a = 0; a < n_atoms; ++a) {
    aoff[a] = (int)atom_off[a];
    for (int64_t j = atom_off[a]; j < atom_off[a + 1]; ++j) orb_atom[j] = a;
  }
  aoff[n_atoms] = n;
  const size_t need = gb_forces_workspace_size(m, p, n_atoms);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
    return fail(GB_EINVAL, "workspace must be a 256-byte aligned device pointer");
  if (workspace_bytes < need) return fail(GB_ENOMEM, "workspace too small: %zu < %zu bytes", workspace_bytes, need);
  std::vector<long long> off(nrhs + 1, 0);
  for (int c = 0; c < nrhs; ++c) {
    const int j = p->rhs_cols[c];
    off[c + 1] = off[c] + (m->h_row_ptr[j + 1] - m->h_row_ptr[j]);
  }
  // packed index of every CSR element's transpose: entry e = (row j, column i)
  // lies in column j; the element (i, j) lies in column i at the position of j in R_i
  const std::vector<int64_t>& rp = m->h_row_ptr;
  std::vector<int32_t> ci(m->nnz);
  GB_CUDA(cudaMemcpy(ci.data(), m->dm.col_idx, 4 * (size_t)m->nnz, cudaMemcpyDeviceToHost));
  std::vector<long long> tp(m->nnz);
  for (int j = 0; j < n; ++j)
    for (int64_t e = rp[j]; e < rp[j + 1]; ++e) {
      const int i = ci[e];
      const int32_t* r0 = ci.data() + rp[i];
      const int32_t* r1 = ci.data() + rp[i + 1];
      const int32_t* hit = std::lower_bound(r0, r1, j);
      if (hit == r1 || *hit != j) return fail(GB_EINVAL, "the pattern is not symmetric");
      tp[e] = off[col_of[i]] + (hit - r0);
    }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(workspace);
  int* d_aoff = reinterpret_cast<int*>(w);
  int* d_atom = reinterpret_cast<int*>(w + align256(4 * ((size_t)n_atoms + 1)));
  int* d_col = reinterpret_cast<int*>(w + align256(4 * ((size_t)n_atoms + 1)) + align256(4 * (size_t)n));
  long long* d_off =
      reinterpret_cast<long long*>(w + align256(4 * ((size_t)n_atoms + 1)) + 2 * align256(4 * (size_t)n));
  GB_CUDA(cudaMemcpyAsync(d_aoff, aoff.data(), 4 * ((size_t)n_atoms + 1), cudaMemcpyHostToDevice, s));
  GB_CUDA(cudaMemcpyAsync(d_atom, orb_atom.data(), 4 * (size_t)n, cudaMemcpyHostToDevice, s));
  GB_CUDA(cudaMemcpyAsync(d_col, col_of.data(), 4 * (size_t)n, cudaMemcpyHostToDevice, s));
  GB_CUDA(cudaMemcpyAsync(d_off, off.data(), 8 * ((size_t)nrhs + 1), cudaMemcpyHostToDevice, s));
  long long* d_tp = reinterpret_cast<long long*>(reinterpret_cast<char*>(d_off) + align256(8 * ((size_t)nrhs + 1)));
  GB_CUDA(cudaMemcpyAsync(d_tp, tp.data(), 8 * (size_t)m->nnz, cudaMemcpyHostToDevice, s));
  const unsigned blocks = (unsigned)(((long long)n_atoms * 32 + 255) / 256);
  forces_kernel<<<blocks, 256, 0, s>>>(m->dm, d_aoff, d_atom, d_col, d_off, d_tp, rho, edm, grad_h, grad_s,
                                       (long long)m->nnz, n_atoms, forces);
  GB_CUDA(cudaGetLastError());
  GB_CUDA(cudaStreamSynchronize(s));  // the host staging vectors are this call's locals
  return GB_OK;
}

}  // extern "C"

// ------------------------------------------------------------ S^-1 terms
// A pole expansion of the Fermi function leaves, besides the resolvents the
// shifted solve forms, multiples of S^-1 (in rho and P^E) and of S^-1 H S^-1
// (in P^E).  gb_add_sinv_terms adds them on the pattern: one team per chunk of
// 32 columns forms X = S^-1 E (E the unit columns), Y = H X and Z = S^-1 Y with
// the FP64 factor, then rho_ij += a X_ij and P^E_ij += b X_ij + c Z_ij on the
// pattern rows of each column; q and E are then recomputed from rho.
namespace {

__global__ void __launch_bounds__(gbk::TPB, 1)
    sinv_terms_kernel(const __grid_constant__ gbk::Args a, const int* __restrict__ cols,
                      const long long* __restrict__ off, int nrhs, double a_rho, double b_edm, double c_shs,
                      double* __restrict__ rho, double* __restrict__ edm, char* __restrict__ scratch,
                      size_t panel_bytes, int* __restrict__ status) {
  __shared__ gbk::Smem sm;
  extern __shared__ __align__(16) char dyn_smem[];
  gbk::team_init(sm, dyn_smem);
  constexpr int W = 32;
  const int c0 = blockIdx.x * W, tid = threadIdx.x;
  const int N4 = 4 * a.m.nb;
  char* base = scratch + (size_t)blockIdx.x * 5 * panel_bytes;
  double2* E = reinterpret_cast<double2*>(base);
  double2* X = reinterpret_cast<double2*>(base + panel_bytes);
  double2* Z = reinterpret_cast<double2*>(base + 2 * panel_bytes);
  double2* t1 = reinterpret_cast<double2*>(base + 3 * panel_bytes);
  double2* t2 = reinterpret_cast<double2*>(base + 4 * panel_bytes);
  if (tid < gbk::WMAX) sm.act[tid] = (tid < W && c0 + tid < nrhs) ? 1 : 0;
  if (tid == 0) sm.inner_count = 0;
  for (size_t e = tid; e < (size_t)N4 * W; e += gbk::TPB) {
    const int row = (int)(e / W), l = (int)(e - (size_t)row * W);
    E[e] = make_double2((c0 + l < nrhs && cols[c0 + l] == row) ? 1.0 : 0.0, 0.0);
  }
  __syncthreads();
  gbk::bc_solve64(a, sm, E, X, t1, t2);  // X = S^-1 E (ends with a barrier)
  for (int it = tid; it < a.m.nb * W; it += gbk::TPB) {  // E <- H X
    const int I = it / W, l = it - I * W;
    double2 acc[4];
    gbk::bsr_row_d(a.m, a.m.hb, X, W, l, I, acc);
#pragma unroll
    for (int r = 0; r < 4; ++r) E[(size_t)(4 * I + r) * W + l] = acc[r];
  }
  __syncthreads();
  gbk::bc_solve64(a, sm, E, Z, t1, t2);  // Z = S^-1 H S^-1 E
  for (int l = 0; l < W && c0 + l < nrhs; ++l) {
    const int c = c0 + l, j = cols[c], e0 = a.m.row_ptr[j], len = a.m.row_ptr[j + 1] - e0;
    for (int t = tid; t < len; t += gbk::TPB) {
      const int i = a.m.col_idx[e0 + t];
      const double x = X[(size_t)i * W + l].x, zv = Z[(size_t)i * W + l].x;
      const long long o = off[c] + t;
      if (rho) rho[o] += a_rho * x;
      if (edm) edm[o] += b_edm * x + c_shs * zv;
    }
  }
  if (tid == 0 && sm.bc_fail) atomicOr(status, gbk::kStTimeout);
}

}  // namespace

extern "C" {

size_t gb_add_sinv_terms_workspace_size(const gb_matrix* m, const gb_solve_params* p) {
  clear_error();
  if (!m || !p || p->nrhs < 1) {
    fail(GB_EINVAL, "NULL argument or no columns");
    return 0;
  }
  const size_t chunks = ((size_t)p->nrhs + 31) / 32, panel = align256(16 * 4 * (size_t)m->nb * 32);
  return align256(4 * (size_t)p->nrhs) + align256(8 * ((size_t)p->nrhs + 1)) + 256 + chunks * 5 * panel;
}

gb_status gb_add_sinv_terms(const gb_matrix* m, const gb_solve_params* p, double a_rho, double b_edm, double c_shs,
                            const gb_outputs* out, void* workspace, size_t workspace_bytes, void* stream) {
  clear_error();
  if (!m || !p || !out || !p->rhs_cols || p->nrhs < 1) return fail(GB_EINVAL, "NULL argument or no columns");
  if (m->dm.bf_bw <= 0) return fail(GB_EINVAL, "no factor: S's half-bandwidth exceeds 63");
  if (check_outputs(out) != GB_OK) return GB_EINVAL;
  const int nrhs = p->nrhs;
  for (int c = 0; c < nrhs; ++c)
    if (p->rhs_cols[c] < 0 || p->rhs_cols[c] >= m->n) return fail(GB_EINVAL, "rhs_cols[%d] out of range", c);
  const size_t need = gb_add_sinv_terms_workspace_size(m, p);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
    return fail(GB_EINVAL, "workspace must be a 256-byte aligned device pointer");
  if (workspace_bytes < need) return fail(GB_ENOMEM, "workspace too small: %zu < %zu bytes", workspace_bytes, need);
  int dev = 0;
  GB_CUDA(cudaGetDevice(&dev));
  if (dev != m->device) return fail(GB_EINVAL, "current device differs from the matrix's device");
  std::vector<long long> off(nrhs + 1, 0);
  for (int c = 0; c < nrhs; ++c) {
    const int j = p->rhs_cols[c];
    off[c + 1] = off[c] + (m->h_row_ptr[j + 1] - m->h_row_ptr[j]);
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(workspace);
  int* d_cols = reinterpret_cast<int*>(w);
  long long* d_off = reinterpret_cast<long long*>(w + align256(4 * (size_t)nrhs));
  int* d_st = reinterpret_cast<int*>(w + align256(4 * (size_t)nrhs) + align256(8 * ((size_t)nrhs + 1)));
  char* scratch = w + align256(4 * (size_t)nrhs) + align256(8 * ((size_t)nrhs + 1)) + 256;
  const size_t panel = align256(16 * 4 * (size_t)m->nb * 32);
  GB_CUDA(cudaMemcpyAsync(d_cols, p->rhs_cols, 4 * (size_t)nrhs, cudaMemcpyHostToDevice, s));
  GB_CUDA(cudaMemcpyAsync(d_off, off.data(), 8 * ((size_t)nrhs + 1), cudaMemcpyHostToDevice, s));
  GB_CUDA(cudaMemsetAsync(d_st, 0, sizeof(int), s));
  GB_CUDA(cudaMemsetAsync(scratch, 0, (size_t)((nrhs + 31) / 32) * 5 * panel, s));
  gbk::Args a;
  std::memset(&a, 0, sizeof a);
  a.m = m->dm;
  a.W = 32;
  a.inner_bchol = 1;
  a.bc_bw_alloc = m->dm.bf_bw;
  const size_t dyn = gbk::dyn_layout(true, 32, true, 0, m->dm.bf_bw).bytes;
  GB_CUDA(cudaFuncSetAttribute(sinv_terms_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
  const unsigned chunks = (unsigned)((nrhs + 31) / 32);
  sinv_terms_kernel<<<chunks, gbk::TPB, dyn, s>>>(a, d_cols, d_off, nrhs, a_rho, b_edm, c_shs, out->rho, out->edm,
                                                   scratch, panel, d_st);
  GB_CUDA(cudaGetLastError());
  if (out->rho && (out->q || out->e_loc)) {
    local_sums_kernel<<<(unsigned)((nrhs + 255) / 256), 256, 0, s>>>(m->dm, d_cols, d_off, nrhs, out->rho, out->q,
                                                                     out->e_loc);
    GB_CUDA(cudaGetLastError());
  }
  int hst = 0;
  GB_CUDA(cudaMemcpyAsync(&hst, d_st, sizeof(int), cudaMemcpyDeviceToHost, s));
  GB_CUDA(cudaStreamSynchronize(s));
  if (hst & gbk::kStTimeout) return fail(GB_ETIMEOUT, "a bounded wait for a staged factor tile gave up");
  return GB_OK;
}

}  // extern "C"

// ------------------------------------------------------------ wavepacket propagation
// i S dc/dt = H c (time in hbar / eV): the transport simulations propagate a
// hole wavepacket with a Schroedinger-type equation (Quantum wavepacket
// dynamics).  One step c <- exp(-i tau S^-1 H) c is a Chebyshev series: with
// A = S^-1 H, spec(A) in [e_min, e_max], b = (e_max + e_min) / 2,
// a = (e_max - e_min) / 2 and A~ = (A - b) / a, the Jacobi-Anger expansion
//   exp(-i tau A) = e^{-i b tau} [J_0(a tau) + 2 sum_{k>=1} (-i)^k J_k(a tau) T_k(A~)]
// with T_{k+1} = 2 A~ T_k - T_{k-1}.  Each term costs one H product and one
// FP64 factor solve; the series stops where |J_k(a tau)| < 1e-17.  One team
// per chunk of W wavepackets runs every step (persistent); W is the smallest
// power of two that spreads the packets over the SMs (at most 32).  Where two or more
// SMs are left for each packet, a cluster of teams shares it (wavepacket_cluster.cuh).
namespace {

constexpr int kWpMaxTerms = 256;

__global__ void __launch_bounds__(gbk::TPB, 1)
    wavepacket_kernel(const __grid_constant__ gbk::Args a, double2* __restrict__ psi, int nwp, int nsteps,
                      const double2* __restrict__ coef, int nterms, double ca, double cb, double2 phase,
                      char* __restrict__ scratch, size_t panel_bytes, int* __restrict__ status) {
  __shared__ gbk::Smem sm;
  extern __shared__ __align__(16) char dyn_smem[];
  gbk::team_init(sm, dyn_smem);
  const int W = a.W;  // columns per team (1 .. 32)
  const int c0 = blockIdx.x * W, tid = threadIdx.x, n = a.m.n;
  const size_t NW = (size_t)4 * a.m.nb * W;
  char* base = scratch + (size_t)blockIdx.x * 7 * panel_bytes;
  double2* P = reinterpret_cast<double2*>(base);
  double2* Tm = reinterpret_cast<double2*>(base + panel_bytes);      // T_{k-1}
  double2* Tk = reinterpret_cast<double2*>(base + 2 * panel_bytes);  // T_k
  double2* Y = reinterpret_cast<double2*>(base + 3 * panel_bytes);
  double2* HX = reinterpret_cast<double2*>(base + 4 * panel_bytes);
  double2* t1 = reinterpret_cast<double2*>(base + 5 * panel_bytes);
  double2* t2 = reinterpret_cast<double2*>(base + 6 * panel_bytes);
  if (tid < gbk::WMAX) sm.act[tid] = (tid < W && c0 + tid < nwp) ? 1 : 0;
  if (tid == 0) sm.inner_count = 0;
  for (size_t e = tid; e < NW; e += gbk::TPB) {  // panel layout: row-major, W columns
    const int row = (int)(e / W), l = (int)(e - (size_t)row * W);
    P[e] = (row < n && c0 + l < nwp) ? psi[(size_t)row * nwp + c0 + l] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  auto cm = [](double2 x, double2 y) { return make_double2(x.x * y.x - x.y * y.y, x.x * y.y + x.y * y.x); };
  // Y <- S^-1 H X (ends with a barrier)
  auto apply_a = [&](const double2* X) {
    for (int it = tid; it < a.m.nb * W; it += gbk::TPB) {
      const int I = it / W, l = it - I * W;
      double2 acc[4];
      gbk::bsr_row_d(a.m, a.m.hb, X, W, l, I, acc);
#pragma unroll
      for (int r = 0; r < 4; ++r) HX[(size_t)(4 * I + r) * W + l] = acc[r];
    }
    __syncthreads();
    gbk::bc_solve64(a, sm, HX, Y, t1, t2);
  };
  for (int step = 0; step < nsteps; ++step) {
    double2* tm = Tm;
    double2* tk = Tk;
    // T_0 = P, accumulate c_0 T_0 into P's replacement at the end (held in Tm / Tk roles)
    for (size_t e = tid; e < NW; e += gbk::TPB) tm[e] = P[e];
    __syncthreads();
    apply_a(tm);  // Y = A T_0
    for (size_t e = tid; e < NW; e += gbk::TPB) {  // T_1 = (A T_0 - b T_0) / a ; P <- c_0 T_0 + c_1 T_1
      const double2 t0 = tm[e];
      const double2 v = make_double2((Y[e].x - cb * t0.x) * ca, (Y[e].y - cb * t0.y) * ca);
      tk[e] = v;
      const double2 s0 = cm(coef[0], t0), s1 = cm(coef[1], v);
      P[e] = make_double2(s0.x + s1.x, s0.y + s1.y);
    }
    __syncthreads();
    for (int k = 2; k < nterms; ++k) {
      apply_a(tk);  // Y = A T_{k-1}
      const double2 ck = coef[k];
      for (size_t e = tid; e < NW; e += gbk::TPB) {  // T_k = 2 (A T_{k-1} - b T_{k-1}) / a - T_{k-2}
        const double2 t1v = tk[e], t0v = tm[e];
        const double2 v = make_double2(2.0 * (Y[e].x - cb * t1v.x) * ca - t0v.x, 2.0 * (Y[e].y - cb * t1v.y) * ca - t0v.y);
        tm[e] = v;  // the slot of T_{k-2} now holds T_k
        const double2 s = cm(ck, v);
        P[e] = make_double2(P[e].x + s.x, P[e].y + s.y);
      }
      __syncthreads();
      double2* sw = tm;  // T_k becomes the current term
      tm = tk;
      tk = sw;
    }
    for (size_t e = tid; e < NW; e += gbk::TPB) P[e] = cm(phase, P[e]);  // e^{-i b tau}
    __syncthreads();
  }
  for (size_t e = tid; e < NW; e += gbk::TPB) {
    const int row = (int)(e / W), l = (int)(e - (size_t)row * W);
    if (row < n && c0 + l < nwp) psi[(size_t)row * nwp + c0 + l] = P[e];
  }
  if (tid == 0 && sm.bc_fail) atomicOr(status, gbk::kStTimeout);
}

// Launches the cluster kernel if clusters of CS for all packets are resident at once; *e:
// the launch's result.
template <int CS, typename... A>
bool wp_cluster(int nwp, cudaStream_t s, cudaError_t* e, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(nwp * CS));
  cfg.blockDim = dim3(gbk::TPB);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = CS;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int resident = 0;
  if (cudaOccupancyMaxActiveClusters(&resident, gbk::wavepacket_cluster_kernel<CS>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (resident < nwp) return false;
  *e = cudaLaunchKernelEx(&cfg, gbk::wavepacket_cluster_kernel<CS>, args...);
  return true;
}

}  // namespace

extern "C" {

static int wp_width(const gb_matrix* m, int nwp) {
  int nsm = 152;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, m->device);
  int w = 1;
  while (w < 32 && (nwp + w - 1) / w > nsm) w <<= 1;
  return w;
}

size_t gb_wavepacket_workspace_size(const gb_matrix* m, int32_t nwp) {
  clear_error();
  if (!m || nwp < 1) {
    fail(GB_EINVAL, "NULL matrix or no wavepackets");
    return 0;
  }
  const int w = wp_width(m, nwp);
  const size_t chunks = ((size_t)nwp + w - 1) / w, panel = align256(16 * 4 * (size_t)m->nb * w);
  return align256(16 * (size_t)kWpMaxTerms) + 256 + chunks * 7 * panel;
}

gb_status gb_wavepacket(const gb_matrix* m, int32_t nwp, void* psi, int32_t nsteps, double tau, double e_min,
                        double e_max, int32_t* nterms_out, void* workspace, size_t workspace_bytes, void* stream) {
  clear_error();
  if (!m || !psi || nwp < 1 || nsteps < 0) return fail(GB_EINVAL, "NULL argument, no wavepackets or nsteps < 0");
  if (misaligned(psi, 16)) return fail(GB_EINVAL, "psi must be 16-byte aligned (complex double)");
  if (m->dm.bf_bw <= 0) return fail(GB_EINVAL, "no factor: S's half-bandwidth exceeds 63");
  if (!(e_max > e_min) || !std::isfinite(e_min) || !std::isfinite(e_max) || !(tau > 0.0) || !std::isfinite(tau))
    return fail(GB_EINVAL, "need e_min < e_max and tau > 0");
  const double ca = 2.0 / (e_max - e_min), cb = 0.5 * (e_max + e_min), z = 0.5 * (e_max - e_min) * tau;
  // Jacobi-Anger coefficients c_0 = J_0(z), c_k = 2 (-i)^k J_k(z) up to |J_k| < 1e-17 past k > z
  std::vector<double2> coef;
  for (int k = 0; k < kWpMaxTerms; ++k) {
    const double j = std::cyl_bessel_j((double)k, z);
    const double mag = k == 0 ? j : 2.0 * j;
    const int r = k & 3;  // (-i)^k = 1, -i, -1, i
    coef.push_back(r == 0 ? make_double2(mag, 0.0)
                   : r == 1 ? make_double2(0.0, -mag)
                   : r == 2 ? make_double2(-mag, 0.0)
                            : make_double2(0.0, mag));
    if (k >= 2 && k > z && std::fabs(j) < 1e-17) break;
  }
  if ((int)coef.size() >= kWpMaxTerms)
    return fail(GB_EINVAL, "(e_max - e_min) tau / 2 = %g needs more than %d terms: take shorter steps", z, kWpMaxTerms);
  const int nterms = (int)coef.size();
  if (nterms_out) *nterms_out = nterms;
  const size_t need = gb_wavepacket_workspace_size(m, nwp);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
    return fail(GB_EINVAL, "workspace must be a 256-byte aligned device pointer");
  if (workspace_bytes < need) return fail(GB_ENOMEM, "workspace too small: %zu < %zu bytes", workspace_bytes, need);
  int dev = 0;
  GB_CUDA(cudaGetDevice(&dev));
  if (dev != m->device) return fail(GB_EINVAL, "current device differs from the matrix's device");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(workspace);
  double2* d_coef = reinterpret_cast<double2*>(w);
  int* d_st = reinterpret_cast<int*>(w + align256(16 * (size_t)kWpMaxTerms));
  char* scratch = w + align256(16 * (size_t)kWpMaxTerms) + 256;
  const int wc = wp_width(m, nwp);
  const size_t panel = align256(16 * 4 * (size_t)m->nb * wc);
  const unsigned chunks = (unsigned)((nwp + wc - 1) / wc);
  GB_CUDA(cudaMemcpyAsync(d_coef, coef.data(), 16 * (size_t)nterms, cudaMemcpyHostToDevice, s));
  GB_CUDA(cudaMemsetAsync(d_st, 0, sizeof(int), s));
  gbk::Args a;
  std::memset(&a, 0, sizeof a);
  a.m = m->dm;
  a.W = wc;
  a.inner_bchol = 1;
  a.bc_bw_alloc = m->dm.bf_bw;
  const double2 phase = make_double2(std::cos(cb * tau), -std::sin(cb * tau));
  auto* x = static_cast<double2*>(psi);
  cudaError_t ce = cudaSuccess;
  auto cluster = [&](auto cs) {
    return wp_cluster<decltype(cs)::value>(nwp, s, &ce, a, x, (int)nwp, (int)nsteps, (const double2*)d_coef, nterms, ca,
                                           cb, phase, scratch, panel, d_st);
  };
  if (wc == 1 && (cluster(std::integral_constant<int, 8>{}) || cluster(std::integral_constant<int, 4>{}) ||
                  cluster(std::integral_constant<int, 2>{}))) {
    GB_CUDA(ce);
  } else {
    const size_t dyn = gbk::dyn_layout(true, wc, true, 0, m->dm.bf_bw).bytes;
    GB_CUDA(cudaFuncSetAttribute(wavepacket_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
    GB_CUDA(cudaMemsetAsync(scratch, 0, (size_t)chunks * 7 * panel, s));
    wavepacket_kernel<<<chunks, gbk::TPB, dyn, s>>>(a, x, nwp, nsteps, d_coef, nterms, ca, cb, phase, scratch, panel,
                                                     d_st);
    GB_CUDA(cudaGetLastError());
  }
  int hst = 0;
  GB_CUDA(cudaMemcpyAsync(&hst, d_st, sizeof(int), cudaMemcpyDeviceToHost, s));
  GB_CUDA(cudaStreamSynchronize(s));
  if (hst & gbk::kStTimeout) return fail(GB_ETIMEOUT, "a bounded wait for a staged factor tile gave up");
  return GB_OK;
}

}  // extern "C"
