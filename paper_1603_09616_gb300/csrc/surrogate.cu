// Learned surrogate for the energy-integrated local outputs (local charge q_j,
// local energy E_j): a per-orbital environment descriptor and a small MLP
// (64 -> 128 -> 128 -> 128 -> 2, GELU, BF16 weights, FP32 accumulation) with
// forward, backward and Adam kernels.  The shifted solver produces the training
// labels and stays the judge (see the Python driver).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

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

constexpr int TILE = 32;

// Y[B x out] = X[B x in] W^T + b, W stored [out x in] in BF16; pre-activation
// kept in P, activation (GELU or identity) in Y.  FP32 accumulation.
__global__ void dense_fwd(const float* __restrict__ X, const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias,
                          int B, int nin, int nout, int act, float* __restrict__ P, float* __restrict__ Y) {
  __shared__ float xs[TILE][TILE + 1];
  __shared__ float ws[TILE][TILE + 1];
  const int row = blockIdx.y * TILE + threadIdx.y;  // sample
  const int col = blockIdx.x * TILE + threadIdx.x;  // output unit
  float acc = 0.f;
  for (int k0 = 0; k0 < nin; k0 += TILE) {
    const int kx = k0 + threadIdx.x;
    xs[threadIdx.y][threadIdx.x] = (row < B && kx < nin) ? X[(size_t)row * nin + kx] : 0.f;
    const int wo = blockIdx.x * TILE + threadIdx.y;  // output unit loaded by this thread row
    ws[threadIdx.y][threadIdx.x] = (wo < nout && kx < nin) ? __bfloat162float(W[(size_t)wo * nin + kx]) : 0.f;
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < TILE; ++k) acc = fmaf(xs[threadIdx.y][k], ws[threadIdx.x][k], acc);
    __syncthreads();
  }
  if (row < B && col < nout) {
    const float p = acc + bias[col];
    P[(size_t)row * nout + col] = p;
    Y[(size_t)row * nout + col] = act ? gelu(p) : p;
  }
}

// G = dY * act'(P) (in place into G), dX[B x in] = G W (BF16 weights)
__global__ void dense_bwd_x(const float* __restrict__ G, const __nv_bfloat16* __restrict__ W, int B, int nin, int nout,
                            float* __restrict__ dX) {
  __shared__ float gs[TILE][TILE + 1];
  __shared__ float ws[TILE][TILE + 1];
  const int row = blockIdx.y * TILE + threadIdx.y;  // sample
  const int col = blockIdx.x * TILE + threadIdx.x;  // input unit
  float acc = 0.f;
  for (int o0 = 0; o0 < nout; o0 += TILE) {
    const int ox = o0 + threadIdx.x;
    gs[threadIdx.y][threadIdx.x] = (row < B && ox < nout) ? G[(size_t)row * nout + ox] : 0.f;
    const int oy = o0 + threadIdx.y;
    const int ic = blockIdx.x * TILE + threadIdx.x;
    ws[threadIdx.y][threadIdx.x] = (oy < nout && ic < nin) ? __bfloat162float(W[(size_t)oy * nin + ic]) : 0.f;
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < TILE; ++k) acc = fmaf(gs[threadIdx.y][k], ws[k][threadIdx.x], acc);
    __syncthreads();
  }
  if (row < B && col < nin) dX[(size_t)row * nin + col] = acc;
}

__global__ void act_grad(float* __restrict__ G, const float* __restrict__ P, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    G[i] *= gelu_grad(P[i]);
}

// dW[out x in] = G^T X (sum over the batch), db = column sums of G; one block
// per (out tile, in tile), batch looped in fixed order (deterministic).
__global__ void dense_bwd_w(const float* __restrict__ G, const float* __restrict__ X, int B, int nin, int nout,
                            float* __restrict__ dW, float* __restrict__ db) {
  __shared__ float gs[TILE][TILE + 1];
  __shared__ float xs[TILE][TILE + 1];
  const int o = blockIdx.y * TILE + threadIdx.y;
  const int i = blockIdx.x * TILE + threadIdx.x;
  float acc = 0.f, accb = 0.f;
  for (int s0 = 0; s0 < B; s0 += TILE) {
    const int sg = s0 + threadIdx.x;
    const int oy = blockIdx.y * TILE + threadIdx.y;
    gs[threadIdx.y][threadIdx.x] = (sg < B && oy < nout) ? G[(size_t)sg * nout + oy] : 0.f;
    const int sx = s0 + threadIdx.y;
    xs[threadIdx.y][threadIdx.x] = (sx < B && i < nin) ? X[(size_t)sx * nin + i] : 0.f;
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < TILE; ++k) {
      acc = fmaf(gs[threadIdx.y][k], xs[k][threadIdx.x], acc);
      accb += gs[threadIdx.y][k];
    }
    __syncthreads();
  }
  if (o < nout && i < nin) dW[(size_t)o * nin + i] = acc;
  if (o < nout && blockIdx.x == 0 && threadIdx.x == 0) db[o] = accb;
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

__global__ void adam_kernel(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                            __nv_bfloat16* __restrict__ wb, size_t n, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    if (wb) wb[i] = __float2bfloat16_rn(wi);
  }
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
  // per layer: pre-activation and activation [batch x width]; plus two gradient buffers
  size_t tot = 0;
  for (int l = 0; l < GB_MLP_LAYERS; ++l) tot += 2 * (size_t)batch * net->dims[l + 1];
  tot += 2 * (size_t)batch * GB_MLP_MAXW;
  tot += 152 * 16;  // loss partials
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
  const float* in = X;
  float* base = ws;
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    const int nin = net->dims[l], nout = net->dims[l + 1];
    float* P = base;
    float* A = base + (size_t)batch * nout;
    base = A + (size_t)batch * nout;
    const bool last = l == GB_MLP_LAYERS - 1;
    dim3 blk(TILE, TILE), grd((nout + TILE - 1) / TILE, (batch + TILE - 1) / TILE);
    dense_fwd<<<grd, blk, 0, s>>>(in, reinterpret_cast<const __nv_bfloat16*>(net->w_bf16[l]), net->b[l], batch, nin,
                                  nout, last ? 0 : 1, P, last ? Y : A);
    in = A;
  }
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
  float* P[GB_MLP_LAYERS];
  float* A[GB_MLP_LAYERS];
  float* base = ws;
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    P[l] = base;
    A[l] = base + (size_t)batch * net->dims[l + 1];
    base = A[l] + (size_t)batch * net->dims[l + 1];
  }
  float* g0 = base;
  float* g1 = base + (size_t)batch * GB_MLP_MAXW;
  cudaMemcpyAsync(g0, dY, sizeof(float) * (size_t)batch * net->dims[GB_MLP_LAYERS], cudaMemcpyDeviceToDevice, s);
  for (int l = GB_MLP_LAYERS - 1; l >= 0; --l) {
    const int nin = net->dims[l], nout = net->dims[l + 1];
    if (l != GB_MLP_LAYERS - 1) {
      const size_t n = (size_t)batch * nout;
      act_grad<<<grid_for(n), 256, 0, s>>>(g0, P[l], n);
    }
    const float* xin = l == 0 ? X : A[l - 1];
    dim3 blk(TILE, TILE);
    dense_bwd_w<<<dim3((nin + TILE - 1) / TILE, (nout + TILE - 1) / TILE), blk, 0, s>>>(g0, xin, batch, nin, nout,
                                                                                          net->gw[l], net->gb[l]);
    if (l > 0) {
      dense_bwd_x<<<dim3((nin + TILE - 1) / TILE, (batch + TILE - 1) / TILE), blk, 0, s>>>(
          g0, reinterpret_cast<const __nv_bfloat16*>(net->w_bf16[l]), batch, nin, nout, g1);
      float* t = g0;
      g0 = g1;
      g1 = t;
    }
  }
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
  for (int l = 0; l < GB_MLP_LAYERS; ++l) {
    if (!net->mw[l] || !net->vw[l] || !net->mb[l] || !net->vb[l]) return gb::fail(GB_EINVAL, "Adam moments are NULL");
    const size_t nw = (size_t)net->dims[l] * net->dims[l + 1], nb = net->dims[l + 1];
    adam_kernel<<<grid_for(nw), 256, 0, s>>>(net->w[l], net->gw[l], net->mw[l], net->vw[l],
                                             reinterpret_cast<__nv_bfloat16*>(net->w_bf16[l]), nw, lr, beta1, beta2,
                                             eps, c1, c2);
    adam_kernel<<<grid_for(nb), 256, 0, s>>>(net->b[l], net->gb[l], net->mb[l], net->vb[l], nullptr, nb, lr, beta1,
                                             beta2, eps, c1, c2);
  }
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
