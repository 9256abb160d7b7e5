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
// activations backward, and the weight gradients of all layers.  The 0.5 GFLOP of a
// training step at batch 2048 are 1 us of tensor cores; what counts is launches and
// latency, so a block takes 16 samples through every layer with the activations in
// shared memory.
//
// FP32 accuracy on BF16 MMAs: an activation (or gradient) is the sum of three BF16
// values, its 24 bits, and the weights are BF16 already, so three exact products
// with FP32 accumulation take the place of one FP32 product.
constexpr int kMlpThreads = 512;
constexpr int kRows = 16, kPad = GB_MLP_MAXW + 8;  // samples per block; row pitch of a plane (bank-conflict free)

struct Net {
  int dims[GB_MLP_LAYERS + 1];
  const __nv_bfloat16* wb[GB_MLP_LAYERS];
  const float* b[GB_MLP_LAYERS];
};
// Where the workspace keeps, per layer, the pre-activation P, the activation A and
// the gradient G of P, all [batch][width].
struct Acts {
  float *P[GB_MLP_LAYERS], *A[GB_MLP_LAYERS], *G[GB_MLP_LAYERS];
  float* part;  // weight-gradient partials
};

struct Planes {
  __nv_bfloat16 v[3][kRows][kPad];
};
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void ldsm2(uint32_t& r0, uint32_t& r1, const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
               : "=r"(r0), "=r"(r1)
               : "r"((uint32_t)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void ldsm2_trans(uint32_t& r0, uint32_t& r1, const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
               : "=r"(r0), "=r"(r1)
               : "r"((uint32_t)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// A fragment of plane p, columns 16 kk ..: lane l names row l % 16, column half l / 16.
__device__ __forceinline__ const void* a_row(const Planes& s, int p, int kk, int lane) {
  return &s.v[p][lane & 15][16 * kk + 8 * (lane >> 4)];
}

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
__device__ __forceinline__ float2 load2(const float* p, bool pair, bool in0, bool in1) {
  if (pair && in1) return *reinterpret_cast<const float2*>(p);
  return make_float2(in0 ? p[0] : 0.f, in1 ? p[1] : 0.f);
}
__device__ __forceinline__ void store2(float* p, bool pair, bool in0, bool in1, float2 v) {
  if (pair && in1) {
    *reinterpret_cast<float2*>(p) = v;
  } else {
    if (in0) p[0] = v.x;
    if (in1) p[1] = v.y;
  }
}
__device__ __forceinline__ bool pairs_ok(const float* p, int width) {
  return (width & 1) == 0 && (reinterpret_cast<uintptr_t>(p) & 7) == 0;
}

// All of a network's weights stay in shared memory (115 KB for the widest one's four
// layers with the activations: one block per SM, which is all a batch of 2048 gives).
// w[l]: layer l, rows [dims[l+1]] x kPad, packed one after the other.
struct MlpSmem {
  Planes x[2];
  __nv_bfloat16 w[1][kPad];
};
__host__ __device__ inline int mlp_rows(const Net& n, int l) { return (n.dims[l + 1] + 15) & ~15; }
size_t mlp_smem(const Net& n) {
  size_t rows = 0;
  for (int l = 0; l < GB_MLP_LAYERS; ++l) rows += mlp_rows(n, l);
  return sizeof(Planes) * 2 + rows * kPad * sizeof(__nv_bfloat16);
}

// One thread's 2 x 2 outputs of its warp's 16 x 8 tile: rows g, g + 8, columns u, u + 1.
// acc: the three planes' sums, the head's in two chains (the tensor cores truncate).
__device__ __forceinline__ float2 tile_row(const float (&d)[4][4], int h) {
  return make_float2((d[0][2 * h] + d[3][2 * h]) + (d[1][2 * h] + d[2][2 * h]),
                     (d[0][2 * h + 1] + d[3][2 * h + 1]) + (d[1][2 * h + 1] + d[2][2 * h + 1]));
}
__device__ __forceinline__ void split3x2(Planes& p, int r, int k, float2 x) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(x.x, x.y);
  const float2 fa = __bfloat1622float2(a), y = make_float2(x.x - fa.x, x.y - fa.y);
  const __nv_bfloat162 b = __floats2bfloat162_rn(y.x, y.y);
  const float2 fb = __bfloat1622float2(b);
  *reinterpret_cast<__nv_bfloat162*>(&p.v[0][r][k]) = a;
  *reinterpret_cast<__nv_bfloat162*>(&p.v[1][r][k]) = b;
  *reinterpret_cast<__nv_bfloat162*>(&p.v[2][r][k]) = __floats2bfloat162_rn(y.x - fb.x, y.y - fb.y);
}
// acc += the 16 samples' planes times the warp's eight columns of B; kk: 16-wide steps.
// TRANS: B is stored [k][column], else [column][k].
template <bool TRANS>
__device__ __forceinline__ void tile_mma(float (&d)[4][4], const Planes& in, const __nv_bfloat16 (*w)[kPad], int steps,
                                         int col0, int lane) {
#pragma unroll 2
  for (int kk = 0; kk < steps; ++kk) {
    uint32_t a[3][4], b0, b1;
#pragma unroll
    for (int p = 0; p < 3; ++p) ldsm4(a[p], a_row(in, p, kk, lane));
    if (TRANS)
      ldsm2_trans(b0, b1, &w[16 * kk + (lane & 15)][col0]);
    else
      ldsm2(b0, b1, &w[col0 + (lane & 7)][16 * kk + 8 * ((lane >> 3) & 1)]);
    mma_bf16(kk & 1 ? d[3] : d[0], a[0], b0, b1);
    mma_bf16(d[1], a[1], b0, b1);
    mma_bf16(d[2], a[2], b0, b1);
  }
}

// Every layer of 16 samples: P = A_prev W^T + b, A = gelu(P) (the last layer: Y = P).
// Warp w forms units 8 w .. 8 w + 7.  Batch 2048: 128 blocks, one wave; bound by the
// latency of four dependent layers (fetch of the weights, MMAs, GELU, barrier).
// Four launches of 32 x 32 FP32 tiles took 47 us.
__global__ void __launch_bounds__(kMlpThreads) mlp_fwd(const Net net, const float* __restrict__ X, int B, Acts ws,
                                                       float* __restrict__ Y) {
  extern __shared__ __align__(16) char mlp_sm[];
  MlpSmem& sm = *reinterpret_cast<MlpSmem*>(mlp_sm);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int row0 = blockIdx.x * kRows, u = 8 * warp + 2 * t;
  {
    int at = 0;
#pragma unroll
    for (int l = 0; l < GB_MLP_LAYERS; ++l) {
      stage_w(net.wb[l], net.dims[l + 1], net.dims[l], sm.w + at);
      at += mlp_rows(net, l);
    }
    const int nin = net.dims[0], kp = (nin + 15) & ~15;
    const bool pair = pairs_ok(X, nin);
    for (int e = tid; e < kRows * kp / 2; e += kMlpThreads) {
      const int r = 2 * e / kp, k = 2 * e - r * kp;
      const bool in = row0 + r < B;
      split3x2(sm.x[0], r, k, load2(X + (size_t)(row0 + r) * nin + k, pair, in && k < nin, in && k + 1 < nin));
    }
  }
  int at = 0;
#pragma unroll
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    const int nin = net.dims[l], nout = net.dims[l + 1], np = (nout + 15) & ~15;
    const bool last = l == GB_MLP_LAYERS - 1, in0 = u < nout, in1 = u + 1 < nout;
    const float2 bias = make_float2(in0 ? net.b[l][u] : 0.f, in1 ? net.b[l][u + 1] : 0.f);
    wait_w(GB_MLP_LAYERS - 1 - l);
    __syncthreads();
    if (8 * warp < np) {
      float d[4][4] = {};
      tile_mma<false>(d, sm.x[l & 1], sm.w + at, (nin + 15) / 16, 8 * warp, lane);
      float* out = last ? Y : ws.A[l];
      const bool pp = pairs_ok(ws.P[l], nout), po = pairs_ok(out, nout);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = g + 8 * h;
        const size_t o = (size_t)(row0 + r) * nout + u;
        const bool in = row0 + r < B;
        float2 p = tile_row(d, h);
        p.x += bias.x;
        p.y += bias.y;
        const float2 y = last ? p : make_float2(in0 ? gelu(p.x) : 0.f, in1 ? gelu(p.y) : 0.f);
        store2(ws.P[l] + o, pp, in && in0, in && in1, p);
        store2(out + o, po, in && in0, in && in1, y);
        if (!last) split3x2(sm.x[(l + 1) & 1], r, u, y);
      }
    }
    at += mlp_rows(net, l);
  }
}

// Gradients of every layer's pre-activations for 16 samples: G of the last layer is
// dY; G_{l-1} = (G_l W_l) gelu'(P_{l-1}).  Warp w forms columns 8 w .. 8 w + 7.
__global__ void __launch_bounds__(kMlpThreads) mlp_bwd_x(const Net net, const float* __restrict__ dY, int B, Acts ws) {
  extern __shared__ __align__(16) char mlp_sm[];
  MlpSmem& sm = *reinterpret_cast<MlpSmem*>(mlp_sm);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int row0 = blockIdx.x * kRows, u = 8 * warp + 2 * t;
  {
    int at = 0;
#pragma unroll
    for (int l = GB_MLP_LAYERS - 1; l > 0; --l) {
      stage_w(net.wb[l], net.dims[l + 1], net.dims[l], sm.w + at);
      at += mlp_rows(net, l);
    }
    const int n = net.dims[GB_MLP_LAYERS], kp = (n + 15) & ~15;
    for (int e = tid; e < kRows * kp / 2; e += kMlpThreads) {
      const int r = 2 * e / kp, k = 2 * e - r * kp;
      const bool in = row0 + r < B;
      split3x2(sm.x[0], r, k, load2(dY + (size_t)(row0 + r) * n + k, false, in && k < n, in && k + 1 < n));
    }
  }
  int at = 0;
#pragma unroll
  for (int l = GB_MLP_LAYERS - 1, it = 0; l > 0; --l, ++it) {
    const int nin = net.dims[l], nout = net.dims[l + 1], np = (nin + 15) & ~15;
    const bool in0 = u < nin, in1 = u + 1 < nin, pp = pairs_ok(ws.P[l - 1], nin), pg = pairs_ok(ws.G[l - 1], nin);
    float2 pre[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const bool in = row0 + g + 8 * h < B;
      pre[h] = load2(ws.P[l - 1] + (size_t)(row0 + g + 8 * h) * nin + u, pp, in && in0, in && in1);
    }
    wait_w(GB_MLP_LAYERS - 2 - it);
    __syncthreads();
    if (8 * warp < np) {
      float d[4][4] = {};
      tile_mma<true>(d, sm.x[it & 1], sm.w + at, (nout + 15) / 16, 8 * warp, lane);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = g + 8 * h;
        const bool in = row0 + r < B;
        float2 v = tile_row(d, h);
        v.x = in && in0 ? v.x * gelu_grad(pre[h].x) : 0.f;
        v.y = in && in1 ? v.y * gelu_grad(pre[h].y) : 0.f;
        store2(ws.G[l - 1] + (size_t)(row0 + r) * nin + u, pg, in && in0, in && in1, v);
        if (l > 1) split3x2(sm.x[(it + 1) & 1], r, u, v);
      }
    }
    at += mlp_rows(net, l);
  }
}

// dW_l = G_l^T A_{l-1} and db_l = column sums of G_l, over one slice of the batch and
// one 64 x 64 tile of one layer (blockIdx.x: the layers' tiles in order), in FP32 on
// the FMA pipes: both operands are FP32, and 84 M products are 2.4 us of the chip.
// Slices give the 12 tiles of the 64-128-128-128-2 network enough blocks; their
// partials are added in order by mlp_bwd_sum (one slice: written in place).
struct GradOut {
  float *gw[GB_MLP_LAYERS], *gb[GB_MLP_LAYERS];
};
__host__ __device__ inline int mlp_slices(int batch) {  // of at least 128 samples, 32 at most
  return batch <= 128 ? 1 : (batch >= 4096 ? 32 : (batch + 127) / 128);
}
__global__ void __launch_bounds__(256) mlp_bwd_w(const Net net, const float* __restrict__ X,
                                                 const float* __restrict__ dY, int B, Acts ws, GradOut out,
                                                 size_t stride) {
  constexpr int KC = 32;  // samples per step, the next step's fetched meanwhile
  __shared__ __align__(16) float gs[KC][68];
  __shared__ __align__(16) float xs[KC][68];
  // the tile's layer (unrolled: the parameters' arrays are not copied to be indexed)
  int tile = blockIdx.x, nin = 0, nout = 0;
  size_t at = 0, next = 0;
  const float *G = nullptr, *A = nullptr;
  float *dw = nullptr, *db = nullptr;
#pragma unroll
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    const int ni = net.dims[l], no = net.dims[l + 1], nt = ((ni + 63) / 64) * ((no + 63) / 64);
    if (tile >= 0 && tile < nt) {
      nin = ni;
      nout = no;
      at = next;
      G = l == GB_MLP_LAYERS - 1 ? dY : ws.G[l];
      A = l == 0 ? X : ws.A[l - 1];
      dw = out.gw[l];
      db = out.gb[l];
      break;
    }
    tile -= nt;
    next += (size_t)no * (ni + 1);
  }
  const int ti = (nin + 63) / 64, o0 = 64 * (tile / ti), i0 = 64 * (tile % ti);
  const int len = ((B + gridDim.y - 1) / gridDim.y + 31) / 32 * 32;
  const int s0 = blockIdx.y * len, s1 = min(B, s0 + len);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  float acc[4][4] = {}, accb[4] = {};
  // thread: rows tid / 16 and + 16 of a step, columns 4 (tid % 16) ..
  const bool gq4 = (nout & 3) == 0 && (reinterpret_cast<uintptr_t>(G) & 15) == 0;
  const bool xq4 = (nin & 3) == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  auto fetch = [&](const float* M, int width, bool quad, int row, int c) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row < s1) {
      const float* p = M + (size_t)row * width + c;
      if (quad) {
        if (c < width) v = *reinterpret_cast<const float4*>(p);
      } else {
        if (c < width) v.x = p[0];
        if (c + 1 < width) v.y = p[1];
        if (c + 2 < width) v.z = p[2];
        if (c + 3 < width) v.w = p[3];
      }
    }
    return v;
  };
  float4 gn[2], xn[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    gn[q] = fetch(G, nout, gq4, s0 + ty + 16 * q, o0 + 4 * tx);
    xn[q] = fetch(A, nin, xq4, s0 + ty + 16 * q, i0 + 4 * tx);
  }
  for (int s = s0; s < s1; s += KC) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      *reinterpret_cast<float4*>(&gs[ty + 16 * q][4 * tx]) = gn[q];
      *reinterpret_cast<float4*>(&xs[ty + 16 * q][4 * tx]) = xn[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      gn[q] = fetch(G, nout, gq4, s + KC + ty + 16 * q, o0 + 4 * tx);
      xn[q] = fetch(A, nin, xq4, s + KC + ty + 16 * q, i0 + 4 * tx);
    }
#pragma unroll 8
    for (int r = 0; r < KC; ++r) {
      const float4 gv = *reinterpret_cast<const float4*>(&gs[r][4 * ty]);
      const float4 xv = *reinterpret_cast<const float4*>(&xs[r][4 * tx]);
      const float gq[4] = {gv.x, gv.y, gv.z, gv.w}, xq[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        accb[i] += gq[i];
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(gq[i], xq[j], acc[i][j]);
      }
    }
    __syncthreads();
  }
  if (gridDim.y > 1) {
    dw = ws.part + blockIdx.y * stride + at;
    db = dw + (size_t)nout * nin;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int o = o0 + 4 * ty + i;
    if (o >= nout) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (i0 + 4 * tx + j < nin) dw[(size_t)o * nin + i0 + 4 * tx + j] = acc[i][j];
    if (i0 == 0 && tx == 0) db[o] = accb[i];
  }
}
__global__ void __launch_bounds__(256) mlp_bwd_sum(const Net net, const float* __restrict__ part, int slices,
                                                   size_t stride, GradOut out) {
  size_t i = blockIdx.x * 256ull + threadIdx.x;
  if (i >= stride) return;
  float s = 0.f;
#pragma unroll 8
  for (int q = 0; q < slices; ++q) s += part[q * stride + i];
#pragma unroll
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    const size_t nw = (size_t)net.dims[l + 1] * net.dims[l], nb = net.dims[l + 1];
    if (i < nw) {
      out.gw[l][i] = s;
      return;
    }
    i -= nw;
    if (i < nb) {
      out.gb[l][i] = s;
      return;
    }
    i -= nb;
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

// Parameters of the network, and what the kernels need of it and of a workspace.
size_t params(const gb_mlp* net) {
  size_t n = 0;
  for (int l = 0; l < GB_MLP_LAYERS; ++l) n += (size_t)net->dims[l + 1] * (net->dims[l] + 1);
  return n;
}
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
  a.part = ws;
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
  // per layer: pre-activation, activation and gradient [batch x width]; then the
  // partial weight gradients of the batch's slices
  size_t tot = 0;
  for (int l = 0; l < GB_MLP_LAYERS; ++l) tot += 3 * (size_t)batch * net->dims[l + 1];
  return (tot + mlp_slices(batch) * params(net)) * sizeof(float);
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
    tiles += (unsigned)(((net->dims[l] + 63) / 64) * ((net->dims[l + 1] + 63) / 64));
  }
  const size_t stride = params(net);
  const int slices = mlp_slices(batch);
  mlp_bwd_w<<<dim3(tiles, (unsigned)slices), 256, 0, s>>>(n, X, dY, batch, a, out, stride);
  if (slices > 1) mlp_bwd_sum<<<(unsigned)((stride + 255) / 256), 256, 0, s>>>(n, a.part, slices, stride, out);
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
