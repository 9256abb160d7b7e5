// Learned surrogate for the energy-integrated local outputs (local charge q_j,
// local energy E_j): a per-orbital environment descriptor and a small MLP
// (64 -> 128 -> 128 -> 128 -> 2, GELU, BF16 weights, FP32 accumulation) with
// forward, backward and Adam kernels.  The shifted solver produces the training
// labels and stays the judge (see the Python driver).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "../../include/gbgreen_surrogate.h"
#include "gb_internal.h"
#include "kernels.cuh"

namespace gb {
const gbk::DevMat* devmat_of(const gb_matrix* m);  // the matrix's device view (solver.cu)
}

namespace {

constexpr int kDesc = 64;
constexpr float kRc = 0.5f;       // nm, descriptor cutoff
constexpr float kRbfW = 0.03f;    // nm, radial Gaussian width

__device__ __forceinline__ float cutoff_fn(float r) { return r < kRc ? 0.5f * (cospif(r / kRc) + 1.0f) : 0.0f; }

// One warp per orbital j.  Features (all from the pattern row j, whose
// orbitals belong to the atoms within the interaction cutoff):
//   0-15  radial Gaussians (centres 0.1..0.5 nm) over carbon neighbour atoms
//   16-31 the same over hydrogen neighbour atoms
//   32-39 angular: per radial shell (4 shells of 0.125 nm) the squared norm of
//         the cutoff-weighted dipole (l = 1) and traceless quadrupole (l = 2)
//         of the neighbour directions
//   40-41 own species one-hot, 42-45 orbital slot one-hot
//   46 H_jj, 47 S_jj
//   48-55 neighbour onsite energies H_ii in 8 Gaussian bins on [-3, 3] eV,
//         weighted by H_ji^2
//   56 sum H_ji^2, 57 sum S_ji^2, 58 sum H_ji S_ji, 59 sum H_ji^2 H_ii,
//   60 sum |H_ji|, 61 |R_j| / 100, 62 sum S_ji H_ii (all over i != j), 63 = 1
//
// The lanes take the row's entries (coalesced) and sum the coupling features in a
// shuffle tree; each neighbour atom a lane finds is then shown to the whole warp,
// lane t adding to radial feature t and lanes 0 .. 8 to the nine angular moments.
// A row has ~126 entries and ~45 neighbour atoms: bound by issue, not by memory
// (3420 orbitals, 20 bytes an entry: under 2 us of HBM).  One thread per orbital
// with its 64 features in local memory and a search for every H_ii took 710 us for
// 3420 orbitals (27 blocks of 128 threads).
__global__ void __launch_bounds__(256)
    descriptor_kernel(const gbk::DevMat m, const float* __restrict__ pos, const int* __restrict__ orb_atom,
                      const int* __restrict__ atom_first, const int* __restrict__ species, float* __restrict__ out) {
  const int j = (int)((blockIdx.x * 256LL + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (j >= m.n) return;  // uniform per warp
  const int a = orb_atom[j];
  const float ax = pos[3 * a], ay = pos[3 * a + 1], az = pos[3 * a + 2];
  const int lo = m.row_ptr[j], hi = m.row_ptr[j + 1];
  float* o = out + (size_t)j * kDesc;
  float bin[8] = {}, sum[6] = {};  // sum: features 56 .. 60 and 62
  float rad = 0.f, mom[4] = {}, hjj = 0.f, sjj = 0.f;
  const float mu = 0.1f + 0.4f * (lane & 15) / 15.0f;
  for (int e0 = lo; e0 < hi; e0 += 32) {
    const int e = e0 + lane;
    bool atom = false;
    float r = 0.f, w = 0.f, ux = 0.f, uy = 0.f, uz = 0.f;
    int code = 0;  // species, shell
    if (e < hi) {
      const int i = m.col_idx[e];
      const double hji = m.h_val[e], sji = m.s_val[e];
      if (i == j) {
        hjj = (float)hji;
        sjj = (float)sji;
      } else {
        const int b = orb_atom[i];
        const float hii = m.h_diag[i], h2 = (float)(hji * hji);
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const float c = -3.0f + 6.0f * t / 7.0f, d = (hii - c) / 0.75f;
          bin[t] += h2 * __expf(-d * d);
        }
        sum[0] += h2;
        sum[1] += (float)(sji * sji);
        sum[2] += (float)(hji * sji);
        sum[3] += h2 * hii;
        sum[4] += fabsf((float)hji);
        sum[5] += (float)sji * hii;
        if (b != a && i == atom_first[b]) {  // geometric part: each neighbour atom once
          const float dx = pos[3 * b] - ax, dy = pos[3 * b + 1] - ay, dz = pos[3 * b + 2] - az;
          r = sqrtf(dx * dx + dy * dy + dz * dz);
          if (r > 1e-6f && r < kRc) {
            atom = true;
            w = cutoff_fn(r);
            ux = dx / r;
            uy = dy / r;
            uz = dz / r;
            code = (species[b] ? 1 : 0) | min(3, (int)(r / (kRc / 4))) << 1;
          }
        }
      }
    }
    for (unsigned left = __ballot_sync(0xffffffffu, atom); left; left &= left - 1) {
      const int src = __ffs(left) - 1;
      const float rr = __shfl_sync(0xffffffffu, r, src), ww = __shfl_sync(0xffffffffu, w, src);
      const float x = __shfl_sync(0xffffffffu, ux, src), y = __shfl_sync(0xffffffffu, uy, src);
      const float z = __shfl_sync(0xffffffffu, uz, src);
      const int cd = __shfl_sync(0xffffffffu, code, src);
      const float d = (rr - mu) / kRbfW, g = ww * __expf(-d * d);
      if ((lane >> 4) == (cd & 1)) rad += g;
      // lanes 0 .. 2: dipole, 3 .. 8: quadrupole xx yy zz xy xz yz
      const float p = lane == 0 || lane == 3 || lane == 6 || lane == 7 ? x : (lane == 2 || lane == 5 ? z : y);
      const float q = lane < 3 ? 1.f : (lane == 3 ? x : (lane == 4 || lane == 6 ? y : z));
      const float v = ww * (p * q - (lane >= 3 && lane < 6 ? 1.0f / 3 : 0.f));
      const int sh = cd >> 1;
#pragma unroll
      for (int s = 0; s < 4; ++s) mom[s] += s == sh ? v : 0.f;
    }
  }
#pragma unroll
  for (int k = 16; k > 0; k >>= 1) {
#pragma unroll
    for (int t = 0; t < 8; ++t) bin[t] += __shfl_xor_sync(0xffffffffu, bin[t], k);
#pragma unroll
    for (int t = 0; t < 6; ++t) sum[t] += __shfl_xor_sync(0xffffffffu, sum[t], k);
    hjj += __shfl_xor_sync(0xffffffffu, hjj, k);  // one lane has the diagonal entry
    sjj += __shfl_xor_sync(0xffffffffu, sjj, k);
  }
  o[lane] = rad;
#pragma unroll
  for (int s = 0; s < 4; ++s) {  // squared norms: moments 0 .. 2, and 3 .. 8 (off-diagonal ones twice)
    const float v = lane < 9 ? mom[s] * mom[s] * (lane >= 6 ? 2.f : 1.f) : 0.f;
    float dip = lane < 3 ? v : 0.f, quad = lane < 3 ? 0.f : v;
#pragma unroll
    for (int k = 8; k > 0; k >>= 1) {
      dip += __shfl_xor_sync(0xffffffffu, dip, k);
      quad += __shfl_xor_sync(0xffffffffu, quad, k);
    }
    if (lane == 0) {
      o[32 + 2 * s] = dip;
      o[33 + 2 * s] = quad;
    }
  }
  if (lane < 6) o[40 + lane] = lane == (species[a] ? 1 : 0) || lane == 2 + min(3, j - atom_first[a]) ? 1.f : 0.f;
  if (lane == 0) {
    o[46] = hjj;
    o[47] = sjj;
#pragma unroll
    for (int t = 0; t < 8; ++t) o[48 + t] = bin[t];
#pragma unroll
    for (int t = 0; t < 5; ++t) o[56 + t] = sum[t];
    o[61] = (hi - lo) / 100.0f;
    o[62] = sum[5];
    o[63] = 1.f;
  }
}

// ------------------------------------------------------------ MLP kernels
__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float x) {
  const float cdf = 0.5f * (1.0f + erff(x * 0.70710678118654752f));
  const float pdf = 0.39894228040143268f * __expf(-0.5f * x * x);
  return cdf + x * pdf;
}

// The network runs in three kernels: all four layers forward, the gradients of the
// activations backward, and the weight gradients of all layers.  The 0.25 G products
// of a training step at batch 2048 are 6 us of the FP32 pipes; what counts beside them
// is launches and latency, so a block takes 16 samples through every layer with the
// activations in shared memory.
//
// Every product's sum runs over its index in ascending order in one FP32 accumulator.
// Adam's first steps divide a gradient by its own magnitude (beside eps = 1e-8), so a
// bias whose gradient cancels over the batch shows the order of the additions: sums in
// slices, or in the tensor cores' order, are as exact, but moved such a step by 1e-3 of
// the learning rate.  GB300, steps back to back, against three-way BF16 splits on the tensor
// cores with the batch in slices, and against a launch of 32 x 32 tiles for each product:
// batch 512 57 / 64 / 233 us, 2048 73 / 65 / 607, 32,768 834 / 345 / 8382.
constexpr int kMlpThreads = 512;
constexpr int kRows = 16;                  // samples per block
constexpr int kPad = GB_MLP_MAXW + 8;      // row pitch of a weight plane (16 bytes a row more: no bank conflicts)
constexpr int kXPad = GB_MLP_MAXW + 4;     // and of the activations

struct Net {
  int dims[GB_MLP_LAYERS + 1];
  const __nv_bfloat16* wb[GB_MLP_LAYERS];
  const float* b[GB_MLP_LAYERS];
};
// Where the workspace keeps, per layer, the pre-activation P, the activation A and
// the gradient G of P, all [batch][width].
struct Acts {
  float *P[GB_MLP_LAYERS], *A[GB_MLP_LAYERS], *G[GB_MLP_LAYERS];
};

// Weights W [rows][cols] into shared memory, pitch kPad, zero up to multiples of 16;
// asynchronous (one commit group) where the rows are whole 16-byte pieces.
__device__ __forceinline__ void stage_w(const __nv_bfloat16* __restrict__ W, int rows, int cols,
                                        __nv_bfloat16 (*s)[kPad]) {
  const int rp = (rows + 15) & ~15, cp = (cols + 15) & ~15;
  if ((cols & 7) == 0 && (reinterpret_cast<uintptr_t>(W) & 15) == 0) {
    const int c8 = cp / 8;
    for (int e = threadIdx.x; e < rp * c8; e += kMlpThreads) {
      const int r = e / c8, c = 8 * (e - r * c8);
      if (r < rows && c < cols)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(&s[r][c])),
                     "l"(W + (size_t)r * cols + c)
                     : "memory");
      else
        *reinterpret_cast<uint4*>(&s[r][c]) = make_uint4(0, 0, 0, 0);
    }
  } else {
    for (int e = threadIdx.x; e < rp * cp; e += kMlpThreads) {
      const int r = e / cp, c = e - r * cp;
      s[r][c] = r < rows && c < cols ? W[(size_t)r * cols + c] : __float2bfloat16(0.f);
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// Groups are committed in the layers' order: all but the `left` last ones are there.
// A barrier must follow.
__device__ __forceinline__ void wait_w(int left) {
  switch (left) {
    case 0: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
    case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
    case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
    default: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
  }
}
// The 16 samples' rows of M [B][width] into shared memory, zero up to a multiple of 16 columns.
__device__ __forceinline__ void stage_x(const float* __restrict__ M, int row0, int B, int width, float (*s)[kXPad]) {
  const int cp = (width + 15) & ~15;
  for (int e = threadIdx.x; e < kRows * cp; e += kMlpThreads) {
    const int r = e / cp, c = e - r * cp;
    s[r][c] = row0 + r < B && c < width ? M[(size_t)(row0 + r) * width + c] : 0.f;
  }
}
// The two BF16 values of a word, as FP32.
__device__ __forceinline__ float2 bf16_pair(uint32_t v) {
  return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
}

// All of a network's weights stay in shared memory (123 KB for 64-128-128-128-2 and 153 KB
// for the widest network, with the activations: one block per SM, which is all a batch of
// 2048 gives).  w: layer l's rows [dims[l+1] up to 16] x kPad, packed one after the other.
struct MlpSmem {
  float x[2][kRows][kXPad];
  __nv_bfloat16 w[1][kPad];
};
__host__ __device__ inline int mlp_rows(const Net& n, int l) { return (n.dims[l + 1] + 15) & ~15; }
size_t mlp_smem(const Net& n) {
  size_t rows = 0;
  for (int l = 0; l < GB_MLP_LAYERS; ++l) rows += mlp_rows(n, l);
  return sizeof(float) * 2 * kRows * kXPad + rows * kPad * sizeof(__nv_bfloat16);
}

// Every layer of 16 samples: P = A_prev W^T + b, A = gelu(P) (the last layer: Y = P).
// Thread: unit tid % 128 of four samples, eight terms a step (one 16-byte read of the
// unit's weights, the samples' values broadcast to the warp).  Batch 2048: 128 blocks, one
// wave, 17 us a call (four launches of 32 x 32 tiles 47).
__global__ void __launch_bounds__(kMlpThreads) mlp_fwd(const Net net, const float* __restrict__ X, int B, Acts ws,
                                                       float* __restrict__ Y) {
  extern __shared__ __align__(16) char mlp_sm[];
  MlpSmem& sm = *reinterpret_cast<MlpSmem*>(mlp_sm);
  const int u = threadIdx.x % GB_MLP_MAXW, s0 = 4 * (threadIdx.x / GB_MLP_MAXW), row0 = blockIdx.x * kRows;
  {
    int at = 0;
#pragma unroll
    for (int l = 0; l < GB_MLP_LAYERS; ++l) {
      stage_w(net.wb[l], net.dims[l + 1], net.dims[l], sm.w + at);
      at += mlp_rows(net, l);
    }
    stage_x(X, row0, B, net.dims[0], sm.x[0]);
  }
  int at = 0;
#pragma unroll
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    const int nin = net.dims[l], nout = net.dims[l + 1], np = (nout + 15) & ~15;
    const bool last = l == GB_MLP_LAYERS - 1, in = u < nout;
    const float bias = in ? net.b[l][u] : 0.f;
    wait_w(GB_MLP_LAYERS - 1 - l);
    __syncthreads();
    if (u < np) {
      float acc[4] = {};
      const __nv_bfloat16* w = sm.w[at + u];
      const float(*x)[kXPad] = sm.x[l & 1];
#pragma unroll 2
      for (int k = 0; k < nin; k += 8) {
        const uint4 wq = *reinterpret_cast<const uint4*>(w + k);
        const float2 w01 = bf16_pair(wq.x), w23 = bf16_pair(wq.y), w45 = bf16_pair(wq.z), w67 = bf16_pair(wq.w);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const float4 a = *reinterpret_cast<const float4*>(&x[s0 + s][k]);
          const float4 b = *reinterpret_cast<const float4*>(&x[s0 + s][k + 4]);
          acc[s] = fmaf(a.x, w01.x, acc[s]);
          acc[s] = fmaf(a.y, w01.y, acc[s]);
          acc[s] = fmaf(a.z, w23.x, acc[s]);
          acc[s] = fmaf(a.w, w23.y, acc[s]);
          acc[s] = fmaf(b.x, w45.x, acc[s]);
          acc[s] = fmaf(b.y, w45.y, acc[s]);
          acc[s] = fmaf(b.z, w67.x, acc[s]);
          acc[s] = fmaf(b.w, w67.y, acc[s]);
        }
      }
      float* out = last ? Y : ws.A[l];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const float p = acc[s] + bias, y = last ? p : gelu(p);
        if (in && row0 + s0 + s < B) {
          const size_t o = (size_t)(row0 + s0 + s) * nout + u;
          ws.P[l][o] = p;
          out[o] = y;
        }
        if (!last) sm.x[(l + 1) & 1][s0 + s][u] = in ? y : 0.f;
      }
    }
    at += mlp_rows(net, l);
  }
}

// Gradients of every layer's pre-activations for 16 samples: G of the last layer is
// dY; G_{l-1} = (G_l W_l) gelu'(P_{l-1}).  Thread: columns 2 (tid % 64), + 1 of two
// samples, four terms a step.
__global__ void __launch_bounds__(kMlpThreads) mlp_bwd_x(const Net net, const float* __restrict__ dY, int B, Acts ws) {
  extern __shared__ __align__(16) char mlp_sm[];
  MlpSmem& sm = *reinterpret_cast<MlpSmem*>(mlp_sm);
  const int c = 2 * (threadIdx.x % (GB_MLP_MAXW / 2)), s0 = 2 * (threadIdx.x / (GB_MLP_MAXW / 2));
  const int row0 = blockIdx.x * kRows;
  {
    int at = 0;
#pragma unroll
    for (int l = GB_MLP_LAYERS - 1; l > 0; --l) {
      stage_w(net.wb[l], net.dims[l + 1], net.dims[l], sm.w + at);
      at += mlp_rows(net, l);
    }
    stage_x(dY, row0, B, net.dims[GB_MLP_LAYERS], sm.x[0]);
  }
  int at = 0;
#pragma unroll
  for (int l = GB_MLP_LAYERS - 1, it = 0; l > 0; --l, ++it) {
    const int nin = net.dims[l], nout = net.dims[l + 1], np = (nin + 15) & ~15;
    float pre[2][2];
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int j = 0; j < 2; ++j)
        pre[s][j] = row0 + s0 + s < B && c + j < nin ? ws.P[l - 1][(size_t)(row0 + s0 + s) * nin + c + j] : 0.f;
    wait_w(GB_MLP_LAYERS - 2 - it);
    __syncthreads();
    if (c < np) {
      float acc[2][2] = {};
      const __nv_bfloat16(*w)[kPad] = sm.w + at;
      const float(*g)[kXPad] = sm.x[it & 1];
#pragma unroll 4
      for (int o = 0; o < nout; o += 4) {
        float2 wq[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) wq[q] = bf16_pair(*reinterpret_cast<const uint32_t*>(&w[o + q][c]));
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const float4 gv = *reinterpret_cast<const float4*>(&g[s0 + s][o]);
          const float gq[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            acc[s][0] = fmaf(gq[q], wq[q].x, acc[s][0]);
            acc[s][1] = fmaf(gq[q], wq[q].y, acc[s][1]);
          }
        }
      }
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const bool in = row0 + s0 + s < B && c + j < nin;
          const float v = in ? acc[s][j] * gelu_grad(pre[s][j]) : 0.f;
          if (in) ws.G[l - 1][(size_t)(row0 + s0 + s) * nin + c + j] = v;
          if (l > 1) sm.x[(it + 1) & 1][s0 + s][c + j] = v;
        }
    }
    at += mlp_rows(net, l);
  }
}

// dW_l = G_l^T A_{l-1} and db_l = column sums of G_l over the whole batch, for one 16 x 16
// tile of one layer (blockIdx.x: the layers' tiles in order).  Two warps of 2 x 2 outputs a
// thread: a sample is two shared-memory reads and four FMAs, and the 2048 samples of an
// output are a chain of additions whatever is done, so small tiles (168 for the
// 64-128-128-128-2 network: one wave) take the least time.  Samples come through a ring of
// asynchronous copies.
struct GradOut {
  float *gw[GB_MLP_LAYERS], *gb[GB_MLP_LAYERS];
};
constexpr int kGradThreads = 64, kGradTile = 16, kGradStep = 64, kGradRing = 4;
__global__ void __launch_bounds__(kGradThreads) mlp_bwd_w(const Net net, const float* __restrict__ X,
                                                          const float* __restrict__ dY, int B, Acts ws, GradOut out) {
  __shared__ __align__(16) float gs[kGradRing][kGradStep][kGradTile];
  __shared__ __align__(16) float xs[kGradRing][kGradStep][kGradTile];
  // the tile's layer (unrolled: the parameters' arrays are not copied to be indexed)
  int left = blockIdx.x, tile = 0, nin = 0, nout = 0;
  const float *G = nullptr, *A = nullptr;
  float *dw = nullptr, *db = nullptr;
#pragma unroll
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    const int ni = net.dims[l], no = net.dims[l + 1];
    const int nt = ((ni + kGradTile - 1) / kGradTile) * ((no + kGradTile - 1) / kGradTile);
    if (left >= 0 && left < nt) {
      tile = left;
      nin = ni;
      nout = no;
      G = l == GB_MLP_LAYERS - 1 ? dY : ws.G[l];
      A = l == 0 ? X : ws.A[l - 1];
      dw = out.gw[l];
      db = out.gb[l];
    }
    left -= nt;
  }
  const int ti = (nin + kGradTile - 1) / kGradTile, o0 = kGradTile * (tile / ti), i0 = kGradTile * (tile % ti);
  const int tid = threadIdx.x, tx = tid % 8, ty = tid / 8;
  const bool bias = i0 == 0;
  // Rows s .. s + kGradStep - 1 of a matrix's 16 columns; zero beyond the batch and the width.
  auto fetch = [&](const float* __restrict__ M, int width, int c0, int s, float (*dst)[kGradTile]) {
    if ((width & 3) == 0 && (reinterpret_cast<uintptr_t>(M) & 15) == 0) {
#pragma unroll
      for (int q = 0; q < kGradStep * kGradTile / 4 / kGradThreads; ++q) {
        const int e = tid + q * kGradThreads, r = e / (kGradTile / 4), c = 4 * (e % (kGradTile / 4));
        const bool in = s + r < B && c0 + c < width;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(&dst[r][c])),
                     "l"(in ? M + (size_t)(s + r) * width + c0 + c : M), "r"(in ? 16 : 0)
                     : "memory");
      }
    } else {
      for (int e = tid; e < kGradStep * kGradTile; e += kGradThreads) {
        const int r = e / kGradTile, c = e % kGradTile;
        const bool in = s + r < B && c0 + c < width;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(&dst[r][c])),
                     "l"(in ? M + (size_t)(s + r) * width + c0 + c : M), "r"(in ? 4 : 0)
                     : "memory");
      }
    }
  };
  auto issue = [&](int step) {
    const int s = step * kGradStep;
    if (s < B) {
      fetch(G, nout, o0, s, gs[step % kGradRing]);
      fetch(A, nin, i0, s, xs[step % kGradRing]);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int q = 0; q < kGradRing - 1; ++q) issue(q);
  float acc[2][2] = {}, accb[2] = {};
  for (int step = 0; step * kGradStep < B; ++step) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kGradRing - 2) : "memory");
    __syncthreads();  // step's samples are there; the buffer of step - 1 is free
    issue(step + kGradRing - 1);
    const float(*g)[kGradTile] = gs[step % kGradRing];
    const float(*x)[kGradTile] = xs[step % kGradRing];
#pragma unroll 8
    for (int r = 0; r < kGradStep; ++r) {
      const float2 gv = *reinterpret_cast<const float2*>(&g[r][2 * ty]);
      const float2 xv = *reinterpret_cast<const float2*>(&x[r][2 * tx]);
      acc[0][0] = fmaf(gv.x, xv.x, acc[0][0]);
      acc[0][1] = fmaf(gv.x, xv.y, acc[0][1]);
      acc[1][0] = fmaf(gv.y, xv.x, acc[1][0]);
      acc[1][1] = fmaf(gv.y, xv.y, acc[1][1]);
      if (bias) {
        accb[0] += gv.x;
        accb[1] += gv.y;
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int o = o0 + 2 * ty + i;
    if (o >= nout) continue;
#pragma unroll
    for (int j = 0; j < 2; ++j)
      if (i0 + 2 * tx + j < nin) dw[(size_t)o * nin + i0 + 2 * tx + j] = acc[i][j];
    if (bias && tx == 0) db[o] = accb[i];
  }
}

__global__ void mse_grad(const float* __restrict__ Y, const float* __restrict__ T, size_t n, float scale,
                         float* __restrict__ dY, float* __restrict__ partial) {
  __shared__ float red[256];
  float s = 0.f;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float d = Y[i] - T[i];
    dY[i] = 2.0f * scale * d;
    s += d * d;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = red[0] * scale;
}

// One Adam step on every parameter array (blockIdx.y: weights and biases of the layers).
struct AdamArgs {
  float *w[2 * GB_MLP_LAYERS], *m[2 * GB_MLP_LAYERS], *v[2 * GB_MLP_LAYERS];
  const float* g[2 * GB_MLP_LAYERS];
  __nv_bfloat16* wb[2 * GB_MLP_LAYERS];
  int n[2 * GB_MLP_LAYERS];
};
__global__ void __launch_bounds__(256) adam_kernel(const AdamArgs a, float lr, float b1, float b2, float eps, float c1,
                                                   float c2) {
  const int y = blockIdx.y, i = blockIdx.x * 256 + threadIdx.x;
  if (i >= a.n[y]) return;
  const float gi = a.g[y][i];
  const float mi = b1 * a.m[y][i] + (1.f - b1) * gi;
  const float vi = b2 * a.v[y][i] + (1.f - b2) * gi * gi;
  a.m[y][i] = mi;
  a.v[y][i] = vi;
  const float wi = a.w[y][i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  a.w[y][i] = wi;
  if (a.wb[y]) a.wb[y][i] = __float2bfloat16_rn(wi);
}

__global__ void to_bf16(const float* __restrict__ w, __nv_bfloat16* __restrict__ wb, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    wb[i] = __float2bfloat16_rn(w[i]);
}

__global__ void affine_cols(float* __restrict__ X, size_t n, int cols, const float* __restrict__ scale,
                            const float* __restrict__ shift) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int c = (int)(i % cols);
    X[i] = fmaf(X[i], scale[c], shift[c]);
  }
}

int grid_for(size_t n) { return (int)std::min<size_t>((n + 255) / 256, 152 * 16); }

// What the kernels need of the network and of a workspace.
Net net_of(const gb_mlp* net) {
  Net n{};
  for (int l = 0; l <= GB_MLP_LAYERS; ++l) n.dims[l] = net->dims[l];
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    n.wb[l] = reinterpret_cast<const __nv_bfloat16*>(net->w_bf16[l]);
    n.b[l] = net->b[l];
  }
  return n;
}
Acts acts_of(const gb_mlp* net, int batch, float* ws) {
  Acts a{};
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    const size_t n = (size_t)batch * net->dims[l + 1];
    a.P[l] = ws;
    a.A[l] = ws + n;
    a.G[l] = ws + 2 * n;
    ws += 3 * n;
  }
  return a;
}

}  // namespace

extern "C" {

gb_status gb_descriptors(const gb_matrix* m, int32_t n_atoms, const float* pos, const int32_t* orb_atom,
                         const int32_t* atom_first, const int32_t* species, float* out, void* stream) {
  gb::clear_error();
  if (!m || !pos || !orb_atom || !atom_first || !species || !out || n_atoms < 1)
    return gb::fail(GB_EINVAL, "gb_descriptors: NULL argument or no atoms");
  const gbk::DevMat* dm = gb::devmat_of(m);
  descriptor_kernel<<<(dm->n + 7) / 8, 256, 0, static_cast<cudaStream_t>(stream)>>>(*dm, pos, orb_atom, atom_first,
                                                                                    species, out);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return gb::fail(GB_ECUDA, "descriptor kernel: %s", cudaGetErrorString(e));
  return GB_OK;
}

size_t gb_mlp_workspace_size(const gb_mlp* net, int32_t batch) {
  if (!net || batch < 1) return 0;
  // per layer: pre-activation, activation and gradient [batch x width]
  size_t tot = 0;
  for (int l = 0; l < GB_MLP_LAYERS; ++l) tot += 3 * (size_t)batch * net->dims[l + 1];
  return tot * sizeof(float);
}

static gb_status check_net(const gb_mlp* net) {
  if (!net) return gb::fail(GB_EINVAL, "net is NULL");
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    if (net->dims[l] < 1 || net->dims[l] > GB_MLP_MAXW || net->dims[l + 1] < 1 || net->dims[l + 1] > GB_MLP_MAXW)
      return gb::fail(GB_EINVAL, "layer widths must be in [1, %d]", GB_MLP_MAXW);
    if (!net->w[l] || !net->w_bf16[l] || !net->b[l]) return gb::fail(GB_EINVAL, "layer %d has NULL weights", l);
  }
  return GB_OK;
}

gb_status gb_mlp_forward(const gb_mlp* net, const float* X, int32_t batch, float* Y, float* ws, size_t ws_bytes,
                         void* stream) {
  gb::clear_error();
  gb_status st = check_net(net);
  if (st != GB_OK) return st;
  if (!X || !Y || !ws || batch < 1) return gb::fail(GB_EINVAL, "gb_mlp_forward: bad arguments");
  if (ws_bytes < gb_mlp_workspace_size(net, batch)) return gb::fail(GB_ENOMEM, "MLP workspace too small");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const Net n = net_of(net);
  const size_t sm = mlp_smem(n);
  cudaFuncSetAttribute(mlp_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  mlp_fwd<<<(batch + kRows - 1) / kRows, kMlpThreads, sm, s>>>(n, X, batch, acts_of(net, batch, ws), Y);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return gb::fail(GB_ECUDA, "MLP forward: %s", cudaGetErrorString(e));
  return GB_OK;
}

gb_status gb_mlp_backward(const gb_mlp* net, const float* X, const float* dY, int32_t batch, float* ws,
                          size_t ws_bytes, void* stream) {
  gb::clear_error();
  gb_status st = check_net(net);
  if (st != GB_OK) return st;
  if (!X || !dY || !ws || batch < 1) return gb::fail(GB_EINVAL, "gb_mlp_backward: bad arguments");
  if (ws_bytes < gb_mlp_workspace_size(net, batch)) return gb::fail(GB_ENOMEM, "MLP workspace too small");
  for (int l = 0; l < GB_MLP_LAYERS; ++l)
    if (!net->gw[l] || !net->gb[l]) return gb::fail(GB_EINVAL, "layer %d has NULL gradient buffers", l);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const Net n = net_of(net);
  const Acts a = acts_of(net, batch, ws);
  const size_t sm = mlp_smem(n);
  cudaFuncSetAttribute(mlp_bwd_x, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  mlp_bwd_x<<<(batch + kRows - 1) / kRows, kMlpThreads, sm, s>>>(n, dY, batch, a);
  GradOut out;
  unsigned tiles = 0;
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    out.gw[l] = net->gw[l];
    out.gb[l] = net->gb[l];
    tiles += (unsigned)(((net->dims[l] + kGradTile - 1) / kGradTile) * ((net->dims[l + 1] + kGradTile - 1) / kGradTile));
  }
  mlp_bwd_w<<<tiles, kGradThreads, 0, s>>>(n, X, dY, batch, a, out);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return gb::fail(GB_ECUDA, "MLP backward: %s", cudaGetErrorString(e));
  return GB_OK;
}

gb_status gb_mse_grad(const float* Y, const float* T, int32_t batch, int32_t nout, float* dY, float* partial,
                      int32_t* npartial, void* stream) {
  gb::clear_error();
  if (!Y || !T || !dY || !partial || !npartial || batch < 1 || nout < 1) return gb::fail(GB_EINVAL, "gb_mse_grad: bad arguments");
  const size_t n = (size_t)batch * nout;
  const int g = grid_for(n);
  mse_grad<<<g, 256, 0, static_cast<cudaStream_t>(stream)>>>(Y, T, n, 1.0f / (float)n, dY, partial);
  *npartial = g;
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return gb::fail(GB_ECUDA, "mse kernel: %s", cudaGetErrorString(e));
  return GB_OK;
}

gb_status gb_mlp_adam(gb_mlp* net, float lr, float beta1, float beta2, float eps, int32_t step, void* stream) {
  gb::clear_error();
  gb_status st = check_net(net);
  if (st != GB_OK) return st;
  if (step < 1) return gb::fail(GB_EINVAL, "Adam step counts from 1");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  AdamArgs a{};
  int most = 0;
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    if (!net->mw[l] || !net->vw[l] || !net->mb[l] || !net->vb[l]) return gb::fail(GB_EINVAL, "Adam moments are NULL");
    const int w = 2 * l, b = 2 * l + 1;
    a.w[w] = net->w[l];
    a.g[w] = net->gw[l];
    a.m[w] = net->mw[l];
    a.v[w] = net->vw[l];
    a.wb[w] = reinterpret_cast<__nv_bfloat16*>(net->w_bf16[l]);
    a.n[w] = net->dims[l] * net->dims[l + 1];
    a.w[b] = net->b[l];
    a.g[b] = net->gb[l];
    a.m[b] = net->mb[l];
    a.v[b] = net->vb[l];
    a.n[b] = net->dims[l + 1];
    most = std::max(most, std::max(a.n[w], a.n[b]));
  }
  adam_kernel<<<dim3((unsigned)((most + 255) / 256), 2 * GB_MLP_LAYERS), 256, 0, s>>>(a, lr, beta1, beta2, eps, c1, c2);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return gb::fail(GB_ECUDA, "Adam kernel: %s", cudaGetErrorString(e));
  return GB_OK;
}

gb_status gb_affine_cols(float* X, int32_t rows, int32_t cols, const float* scale, const float* shift,
                         void* stream) {
  gb::clear_error();
  if (!X || !scale || !shift || rows < 0 || cols < 1) return gb::fail(GB_EINVAL, "gb_affine_cols: bad arguments");
  const size_t n = (size_t)rows * cols;
  if (n == 0) return GB_OK;
  affine_cols<<<grid_for(n), 256, 0, static_cast<cudaStream_t>(stream)>>>(X, n, cols, scale, shift);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return gb::fail(GB_ECUDA, "affine kernel: %s", cudaGetErrorString(e));
  return GB_OK;
}

gb_status gb_mlp_sync_bf16(gb_mlp* net, void* stream) {
  gb::clear_error();
  gb_status st = check_net(net);
  if (st != GB_OK) return st;
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    const size_t nw = (size_t)net->dims[l] * net->dims[l + 1];
    to_bf16<<<grid_for(nw), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        net->w[l], reinterpret_cast<__nv_bfloat16*>(net->w_bf16[l]), nw);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return gb::fail(GB_ECUDA, "bf16 copy: %s", cudaGetErrorString(e));
  return GB_OK;
}

}  // extern "C"
