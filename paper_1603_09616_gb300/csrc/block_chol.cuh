// Exact inner solve S x = f with the block-bidiagonal Cholesky factor of S.
//
// The shifted COCG recurrence applies S^{-1} once per outer iteration (and the
// mixed path two or more times, around float-float residuals).  An iterative
// inner solve leaves a relative error of its tolerance in every application,
// and near a spectral gap the shifted residuals amplify that error by ~1e9;
// the factor solve is exact to rounding instead.  For S with half-bandwidth
// bw <= 63 the Cholesky factor L, cut into 64-row blocks, is block lower
// bidiagonal (diagonal blocks D_i, sub-diagonal blocks C_i), and with the
// host-built products E_i = D_i^-1 C_i, F_i = D_i^-T C_{i+1}^T:
//   L y = f   :  t_i = D_i^-1 f_i (every block independent),  y_i = t_i - E_i y_{i-1}
//   L^T x = y :  u_i = D_i^-T y_i (every block independent),  x_i = u_i - F_i x_{i+1}
// The triangular products of all blocks run in parallel; only the band products
// walk the blocks in order.  The mixed path's passes are in factor_passes.cuh.
// The FP64 solve is bound by the FP64 FMA rate and reads its tiles through L2.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "kernels.cuh"

namespace gbk {

template <typename T>
struct CplxOf;
template <>
struct CplxOf<float> {
  using type = float2;
};
template <>
struct CplxOf<double> {
  using type = double2;
};

constexpr int kTileBufs = 3;  // band tiles staged: two in flight ahead of the one in use
constexpr unsigned kRedBytes = TPB_WIDE / 32 * NVMAX * 32 * 8;  // block_reduce's partials

// Dynamic shared memory of a team (host and device agree through this):
//   FP32 factor passes: the tensor-core layouts below (pass_layout, mma_layout);
//   FP64 factor chain: [partials: block_reduce's, or the chain's nks x 64 x
//   (W+1) sums]  [y block: 64 x W], in nchunk chunks of up to two columns;
//   iterative inner solve with its vectors in shared memory: [partials] [g, d, q]
struct DynLayout {
  int nchunk, nks, G;
  unsigned o_red, o_ysm, o_cg, bytes;
};
// The seed recurrence's passes (seed_passes.cuh): [S staged factor tiles][input block x 2][output
// block x 2], blocks of 64 rows x P floats (2 W real columns, padded so that
// the B-fragment loads are free of bank conflicts); S = 3 stages up to W = 8,
// 2 beyond.  A tile holds the 20 triangular fragments and the band fragments
// of a half-bandwidth bw (512 bytes each).  block_reduce's partials alias the
// first stage (the passes and the reductions never overlap).
struct MmaLayout {
  int P, nt, S;
  unsigned stage_floats, o_fin, o_ysm, o_xch, bytes;
};
__host__ __device__ inline MmaLayout mma_layout(int W, int bw) {
  MmaLayout L;
  L.P = 2 * W + 8 > 24 ? 2 * W + 8 : 24;
  L.nt = W >= 4 ? W / 4 : 1;  // n-tiles of 8 real columns
  L.S = W <= 8 ? 3 : 2;
  const int n2 = (bw + 7) / 8 > 8 - (64 - bw) / 8 ? (bw + 7) / 8 : 8 - (64 - bw) / 8;
  L.stage_floats = (unsigned)(20 + 4 * n2) * 128u;
  unsigned off = (unsigned)L.S * L.stage_floats * 4u;
  if (off < kRedBytes) off = kRedBytes;
  off = (off + 127u) & ~127u;
  L.o_fin = off;
  off += 2u * 64u * (unsigned)L.P * 4u;
  L.o_ysm = off;
  off += 2u * 64u * (unsigned)L.P * 4u;
  L.o_xch = off;  // band partials handed from one warp to its partner: 8 tiles x 32 lanes x 4
  off += 8u * 32u * 4u * 4u;
  L.bytes = (off + 127u) & ~127u;
  return L;
}

// Mixed path (factor_passes.cuh): [S staged band tiles][output block x 2, FP16
// head and tail words].  A stage holds the band tile's 4 ne fragment pairs (1 KB
// each); a block's words are kOutWords for each of max(R, 8) columns: 32 row pairs
// and 4 of padding, so that stores and ldmatrix rows hit every bank once.
// block_reduce's partials alias the stages (the passes and the reductions never
// overlap).
constexpr int kOutWords = 36;
struct PassLayout {
  unsigned stage, o_y, bytes;
};
__host__ __device__ inline PassLayout pass_layout(int W, int ne) {
  PassLayout L;
  L.stage = (unsigned)ne * 4096u;
  unsigned off = (unsigned)kTileBufs * L.stage;
  if (off < kRedBytes) off = kRedBytes;
  L.o_y = off;
  off += 2u * 2u * (unsigned)(2 * W > 8 ? 2 * W : 8) * kOutWords * 4u;
  L.bytes = (off + 127u) & ~127u;
  return L;
}

__host__ __device__ inline DynLayout dyn_layout(bool fp64, int W, bool bchol, unsigned cg_bytes, int bw = 63,
                                                bool seed = false) {
  DynLayout L{};
  if (bchol && !fp64) {
    L.o_cg = L.bytes = seed ? mma_layout(W, bw).bytes : pass_layout(W, (bw + 15) / 16).bytes;
    return L;
  }
  unsigned red = kRedBytes, y = 0;
  if (bchol) {  // FP64 chain
    L.G = TPB / 64;
    L.nchunk = W / (W < 2 ? 1 : 2);
    // Slices of k.  Two give four warps even for one column, one per scheduler, which
    // keep its FP64 pipe busy; more only add partial sums (eight: 1024 more additions a
    // block against 1920 FMAs at a half-bandwidth of 15).
    L.nks = L.nchunk >= L.G ? 1 : 2;
    y = 64u * (unsigned)W * 16u;
    const unsigned part = (unsigned)(L.nks * 64 * (W + 1)) * 16u;
    red = red > part ? red : part;
  }
  L.o_ysm = L.o_cg = (red + 127u) & ~127u;
  L.bytes = (L.o_cg + (bchol ? y : cg_bytes) + 127u) & ~127u;
  return L;
}

// ------------------------------------------------------------ TMA bulk copy + mbarrier
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// One thread: expect `bytes` on `bar` and start the copy global -> shared.
// src and dst 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void tma_bulk_g2s(void* dst, const void* src, uint32_t bytes, unsigned long long* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait: gives up after 0.2 s (a tile lands in microseconds) or 2^20
// polls, whichever comes first; the caller records the failure and later
// waits of the launch are skipped.  The clock is read only once a wait has
// lasted some polls: a tile is usually there already.
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long* bar, uint32_t parity) {
  for (int it = 0; it < 16; ++it)
    if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  for (int it = 0; it < (1 << 20); ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if (global_ns() - t0 > 200000000ull) break;
  }
  return false;
}

// ------------------------------------------------------------ element helpers
__device__ __forceinline__ float2 bc_in(const float2* p, size_t e) { return p[e]; }
__device__ __forceinline__ float2 bc_in(const float4* p, size_t e) {  // hi parts of a float-float vector
  const float4 v = p[e];
  return make_float2(v.x, v.z);
}
__device__ __forceinline__ double2 bc_in(const double2* p, size_t e) { return p[e]; }
__device__ __forceinline__ void cfma(double2& acc, double m, double2 v) {
  acc.x = fma(m, v.x, acc.x);
  acc.y = fma(m, v.y, acc.y);
}
__device__ __forceinline__ double2 czero() { return make_double2(0.0, 0.0); }

// ------------------------------------------------------------ triangular pass, FP64
// The triangles of D_i^-1 and D_i^-T for a warp that owns row pairs: lane l takes the
// rows l and 63 - l, whose entries together are 65 for every lane.  Entry j of lane l
// lies at j * 32 + l of the tile: the shorter row's l + 1 entries first, then the
// longer one's, each by ascending k.
constexpr int kTriTile = 65 * 32;
struct TriEntry {
  int row, k;
};
__host__ __device__ __forceinline__ TriEntry tri_entry(bool lower, int lane, int j) {
  if (lower) return j <= lane ? TriEntry{lane, j} : TriEntry{63 - lane, j - lane - 1};
  return j <= lane ? TriEntry{63 - lane, 63 - lane + j} : TriEntry{lane, j - 1};
}

// One warp per (block, column chunk); tiles read through L2.  The FP64 FMA rate bounds
// it (two lanes a clock and SM), so what counts is the FMAs issued: with rows l and
// l + 32 a lane, every warp instruction ran its masked half too, 96 per column and block
// against 65 here (with the chain's two slices: 480 orbitals, all columns, 247.9 ->
// 209.3 ms).  Blocks b0 .. b0 + nblk - 1.  No barrier at the end.
template <bool LOWER, int CWV, typename InT>
__device__ __noinline__ void bc_tri_f64(const Args& a, const Smem& sm, const InT* in, double2* out, int b0,
                                        int nblk) {
  const int W = a.W, N4 = 4 * a.m.nb;
  const int nchunk = W / CWV, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const TriEntry s0 = tri_entry(LOWER, lane, 0), s1 = tri_entry(LOWER, lane, lane + 1);
  for (int task = warp; task < nblk * nchunk; task += NWARP) {
    const int at = task / nchunk, ch = task - at * nchunk, blk = b0 + at, c0 = ch * CWV, base = 64 * blk;
    const double* __restrict__ M = a.m.bft + (size_t)(2 * blk + (LOWER ? 0 : 1)) * kTriTile + lane;
    const int kmax = N4 - base;  // rows of the vector from the block on
    double2 acc[CWV], res[CWV];
#pragma unroll
    for (int c = 0; c < CWV; ++c) acc[c] = res[c] = czero();
    int k = s0.k;
#pragma unroll (CWV == 1 ? 4 : 2)
    for (int j = 0; j < 65; ++j, ++k) {
      if (j == lane + 1) {
        k = s1.k;
#pragma unroll
        for (int c = 0; c < CWV; ++c) {
          res[c] = acc[c];
          acc[c] = czero();
        }
      }
      const double m = __ldg(M + j * 32);
#pragma unroll
      for (int c = 0; c < CWV; ++c)
        cfma(acc[c], m, k < kmax ? bc_in(in, (size_t)(base + k) * W + c0 + c) : czero());
    }
#pragma unroll
    for (int c = 0; c < CWV; ++c) {
      if (!sm.act[c0 + c]) continue;
      if (s0.row < kmax) out[(size_t)(base + s0.row) * W + c0 + c] = res[c];
      if (s1.row < kmax) out[(size_t)(base + s1.row) * W + c0 + c] = acc[c];
    }
  }
}

// ------------------------------------------------------------ the sequential chain, FP64
// FWD: y_0 = t_0, y_i = t_i - E_i y_{i-1} (k over the last bw rows of y_{i-1});
// BWD: x_last = u_last, x_i = u_i - F_i x_{i+1} (k over the first bw rows).
// Thread = (row, column chunk, slice of k); partial sums meet in shared
// memory; the tiles are read through L2 (the FP64 solve is bound by the FP64
// FMA rate).  tin and yout may alias (each element is read, a step ahead,
// before it is written, by the same thread).  Ends with a barrier.
template <int CWV, int PF, bool FWD>
__device__ __noinline__ void bc_chain64(const Args& a, Smem& sm, const double* __restrict__ Mall, const double2* tin,
                                        double2* yout) {
  using C = double2;
  const int W = a.W, N4 = 4 * a.m.nb, nblk = a.m.bf_nblk, bw = a.m.bf_bw, tid = threadIdx.x;
  const DynLayout L = dyn_layout(true, W, true, 0);
  extern __shared__ __align__(16) char bc_dyn[];
  C* red = reinterpret_cast<C*>(bc_dyn + L.o_red);
  C* ysm = reinterpret_cast<C*>(bc_dyn + L.o_ysm);
  const int kbase = FWD ? 64 - bw : 0;
  const int nsteps = nblk - 1;
  auto blk_of = [&](int s) { return FWD ? s : nblk - 1 - s; };  // s = 0: the chain's first block
  {  // first block of the chain
    const int i0 = blk_of(0);
    for (int o = tid; o < 64 * W; o += TPB) {
      const int r = o / W, c = o - r * W, row = 64 * i0 + r;
      const C v = row < N4 ? tin[(size_t)64 * i0 * W + o] : czero();
      ysm[o] = v;
      if (row < N4 && sm.act[c]) yout[(size_t)64 * i0 * W + o] = v;
    }
    __syncthreads();
  }
  const int r0 = tid % 64, g = tid / 64;
  const int nks = L.nks, nchunk = L.nchunk;
  const int len = (bw + nks - 1) / nks;
  C tnext[PF];  // this thread's t values (PF per block), a step ahead of use
  auto load_t = [&](int s) {
    const int i = blk_of(s);
#pragma unroll
    for (int m = 0; m < PF; ++m) {
      const int o = tid + m * TPB;
      const int row = 64 * i + o / W;
      tnext[m] = (s <= nsteps && o < 64 * W && row < N4) ? tin[(size_t)64 * i * W + o] : czero();
    }
  };
  load_t(1);
  for (int s = 1; s <= nsteps; ++s) {
    const int i = blk_of(s);
    C tcur[PF];
#pragma unroll
    for (int m = 0; m < PF; ++m) tcur[m] = tnext[m];
    load_t(s + 1);
    const double* __restrict__ Mt = Mall + (size_t)i * 4096;
    // partial products over this thread's slice of k
    for (int ch = (nks == 1 ? g : g / nks); ch < nchunk; ch += (nks == 1 ? L.G : nchunk)) {
      const int ks = nks == 1 ? 0 : g % nks, c0 = ch * CWV;
      const int kb = kbase + ks * len, ke = min(kb + len, kbase + bw);
      C acc[CWV];
#pragma unroll
      for (int j = 0; j < CWV; ++j) acc[j] = czero();
#pragma unroll 2
      for (int k = kb; k < ke; ++k) {
        const double mv = __ldg(Mt + k * 64 + r0);
#pragma unroll
        for (int j = 0; j < CWV; ++j) cfma(acc[j], mv, ysm[k * W + c0 + j]);
      }
#pragma unroll
      for (int j = 0; j < CWV; ++j) red[((size_t)ks * 64 + r0) * (W + 1) + c0 + j] = acc[j];
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < PF; ++m) {
      const int o = tid + m * TPB;
      if (o >= 64 * W) break;
      const int r = o / W, c = o - r * W, row = 64 * i + r;
      C sacc = czero();
      for (int ks = 0; ks < nks; ++ks) sacc = cadd(sacc, red[((size_t)ks * 64 + r) * (W + 1) + c]);
      const C y = row < N4 ? csub(tcur[m], sacc) : czero();
      ysm[o] = y;
      if (row < N4 && sm.act[c]) yout[(size_t)64 * i * W + o] = y;
    }
    __syncthreads();
  }
}

// x = S^-1 f in FP64 for every active column of the panel.  t1, t2: panel-sized
// scratch vectors (global).  Ends with a barrier.
template <int CWV, int PF>
__device__ void bc_solve_w(const Args& a, Smem& sm, const double2* f, double2* x, double2* t1, double2* t2) {
  const size_t part = (size_t)a.m.bf_nblk * 4096;
  const double* bf = a.m.bf64;
  bc_tri_f64<true, CWV>(a, sm, f, t1, 0, a.m.bf_nblk);
  __syncthreads();
  bc_chain64<CWV, PF, true>(a, sm, bf + 2 * part, t1, t1);
  bc_tri_f64<false, CWV>(a, sm, t1, t2, 0, a.m.bf_nblk);
  __syncthreads();
  bc_chain64<CWV, PF, false>(a, sm, bf + 3 * part, t2, x);
  if (threadIdx.x == 0) ++sm.inner_count;
}

__device__ __forceinline__ void bc_solve64(const Args& a, Smem& sm, const double2* f, double2* x, double2* t1,
                                           double2* t2) {
  static_assert(TPB == 512, "outputs per thread assume 512-thread teams");
  if (a.W == 32)
    bc_solve_w<2, 4>(a, sm, f, x, t1, t2);
  else if (a.W == 16)
    bc_solve_w<2, 2>(a, sm, f, x, t1, t2);
  else if (a.W >= 2)
    bc_solve_w<2, 1>(a, sm, f, x, t1, t2);
  else
    bc_solve_w<1, 1>(a, sm, f, x, t1, t2);
}

}  // namespace gbk

#include "factor_passes.cuh"
#include "dense_inverse.cuh"
#include "seed_passes.cuh"
