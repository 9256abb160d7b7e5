// The mixed path's inner solve where S has no banded factor and few orbitals:
// x = S^-1 f to FP32 accuracy as one product with the inverse.
//
// S^-1 is formed once per matrix, on the device in FP64 (blocked Gauss-Jordan), and
// kept as FP16 head / tail MMA fragments with a power-of-two scale, as the factor's
// tiles are (factor_passes.cuh).  A solve packs the right-hand sides into FP16 heads
// and tails and multiplies: a warp owns 16 rows and every column of the panel, so
// each fragment of the inverse is read once per solve (of up to 16 real columns).  The refinement around it
// (inner_real_factor) is the factor's.
//
// What bounds it: the fragments' bytes through L2, 4 n^2 a solve and team (831 KB at 456
// orbitals), and no chain or barrier inside.  The Chebyshev iteration it replaced there
// reads S and five vectors in each of its some 26 steps an application, with a barrier
// each.  GB300, two 456-orbital bundles, all columns, tol 1e-10: 573 -> 210 ms; one solve
// of 32 shifts, Chebyshev / inverse: 152 orbitals 67 / 27 ms, 684 809 / 333, 1026
// 1672 / 718, 1710 (64 columns) 1944 / 860.
#pragma once

namespace gbk {

// B words of the panel: uint4 {head, head, tail, tail} of lane (column, t) of k-step kk
// at (kk R + column) 4 + t, so that a warp's fragment is 512 consecutive bytes.
template <int MUL>
__device__ __noinline__ void di_pack(const Args& a, const Smem& sm, const float* __restrict__ in,
                                     uint4* __restrict__ words) {
  const int R = 2 * a.W, N4 = 4 * a.m.nb, n = a.m.di_nt * R * 4;
  for (int e = threadIdx.x; e < n; e += tpb()) {
    const int t = e & 3, col = (e >> 2) % R, kk = (e >> 2) / R;
    const float sc = sm.fsc[col];
    float v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {  // the pairs of fx_tri: rows t, t + 8 and t + 4, t + 12
      const int row = 16 * kk + t + 8 * (q & 1) + 4 * (q >> 1);
      v[q] = row < N4 ? in[((size_t)row * R + col) * MUL] * sc : 0.f;
    }
    uint4 w;
    split_f16(v[0], v[1], w.x, w.z);
    split_f16(v[2], v[3], w.y, w.w);
    words[e] = w;
  }
}

// out = un S^-1 (words) for NT tiles of 8 columns from tile n0; DEPTH k-steps of
// fragments in flight (more spill: a team's threads have 64 registers).
template <int NT, int DEPTH>
__device__ __noinline__ void di_product(const Args& a, const Smem& sm, const uint4* __restrict__ words,
                                        float* __restrict__ out, int n0) {
  const int R = 2 * a.W, N4 = 4 * a.m.nb, nt = a.m.di_nt;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  for (int mi = warp; mi < nt; mi += nwarp()) {
    const uint4* __restrict__ A = a.m.di + (size_t)mi * nt * 64 + lane;
    float d0[NT][4], d1[NT][4];
#pragma unroll
    for (int ni = 0; ni < NT; ++ni)
#pragma unroll
      for (int q = 0; q < 4; ++q) d0[ni][q] = d1[ni][q] = 0.f;
    uint4 ah[DEPTH], al[DEPTH];
#pragma unroll
    for (int p = 0; p < DEPTH; ++p) {
      ah[p] = __ldg(A + min(p, nt - 1) * 64);
      al[p] = __ldg(A + min(p, nt - 1) * 64 + 32);
    }
    const uint4* b = words + 32 * n0 + lane;
    for (int k0 = 0; k0 < nt; k0 += DEPTH) {
#pragma unroll
      for (int p = 0; p < DEPTH; ++p, b += R * 4) {  // beyond the last k-step: a fragment again, times zero
        const uint4* next = A + min(k0 + p + DEPTH, nt - 1) * 64;
#pragma unroll
        for (int ni = 0; ni < NT; ++ni) {
          const uint4 w = 8 * (n0 + ni) + g < R && k0 + p < nt ? b[32 * ni] : zero;
          mma_f16(d0[ni], ah[p], w.x, w.y);
          mma_f16(d1[ni], ah[p], w.z, w.w);
          mma_f16(d1[ni], al[p], w.x, w.y);
        }
        ah[p] = __ldg(next);
        al[p] = __ldg(next + 32);
      }
    }
#pragma unroll
    for (int ni = 0; ni < NT; ++ni) {
      const int oc = 8 * (n0 + ni) + 2 * t;
      if (oc >= R) continue;
      const float u0 = sm.fun[oc], u1 = sm.fun[oc + 1];
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int row = 16 * mi + g + 8 * hf;
        if (row < N4)
          *reinterpret_cast<float2*>(out + (size_t)row * R + oc) =
              make_float2(u0 * (d0[ni][2 * hf] + d1[ni][2 * hf]), u1 * (d0[ni][2 * hf + 1] + d1[ni][2 * hf + 1]));
      }
    }
  }
}

// x = S^-1 f: arguments and contract of fx_solve (panels of at most 32 real columns);
// `scratch`: a panel-sized region, 16 N4 W bytes (the words take (N4 + 12) 8 W).
template <typename InT>
__device__ void di_solve(const Args& a, Smem& sm, const InT* f, float2* x, void* scratch) {
  constexpr int MUL = sizeof(InT) == 16 ? 2 : 1;
  const int tid = threadIdx.x;
  if (tid < 2 * a.W) {
    const float m = __uint_as_float(sm.fmax[tid]);
    int ex = 0;
    if (m > 0.f && m < INFINITY) frexpf(m, &ex);
    const int k = m > 0.f ? max(-100, min(100, 13 - ex)) : 0;
    sm.fsc[tid] = ldexpf(1.f, k);
    sm.fun[tid] = ldexpf(1.f, max(-126, min(126, a.m.di_ex - k)));
    sm.fmax[tid] = 0;
  }
  __syncthreads();
  uint4* words = static_cast<uint4*>(scratch);
  float* out = reinterpret_cast<float*>(x);
  di_pack<MUL>(a, sm, reinterpret_cast<const float*>(f), words);
  __syncthreads();
  if (a.W <= 4) {
    di_product<1, 2>(a, sm, words, out, 0);
  } else {
    for (int n0 = 0; 4 * n0 < a.W; n0 += 2) di_product<2, 1>(a, sm, words, out, n0);
  }
  if (tid == 0) ++sm.inner_count;
  __syncthreads();
}

// ------------------------------------------------------------ forming S^-1
// In-place blocked Gauss-Jordan of an SPD matrix (no pivoting needed), 32 x 32 blocks,
// two launches a block step: the pivot's row of blocks, then every block from the old
// matrix into the other buffer (so that no block waits for another).  np: the order,
// a multiple of 32, padded with a unit diagonal.
constexpr int kDiB = 32;

__global__ void __launch_bounds__(256) di_fill_kernel(const DevMat m, double* __restrict__ A, int np) {
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= np) return;
  double* r = A + (size_t)row * np;
  for (int j = lane; j < np; j += 32) r[j] = row >= m.n && j == row ? 1.0 : 0.0;
  __syncwarp();
  if (row < m.n)
    for (int e = m.row_ptr[row] + lane; e < m.row_ptr[row + 1]; e += 32) r[m.col_idx[e]] = m.s_val[e];
}

// R(j) = A(k, k)^-1 A(k, j) for block j = blockIdx.x, R(k) = A(k, k)^-1; every block of
// threads inverts the pivot block for itself (32 steps; a launch of its own would take as
// long).  *bad = 1 where a pivot is not positive (S is not SPD).
__global__ void __launch_bounds__(256) di_pivot_kernel(const double* __restrict__ A, int np, int k,
                                                       double* __restrict__ R, int* __restrict__ bad) {
  __shared__ double s[kDiB][kDiB + 1], X[kDiB][kDiB + 1];
  const int bj = blockIdx.x, j = threadIdx.x & 31, i0 = threadIdx.x >> 5;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const double* row = A + (size_t)(kDiB * k + i0 + 8 * r) * np;
    s[i0 + 8 * r][j] = row[kDiB * k + j];
    X[i0 + 8 * r][j] = row[kDiB * bj + j];
  }
  __syncthreads();
  for (int p = 0; p < kDiB; ++p) {
    const double piv = s[p][p], ip = 1.0 / piv, pj = s[p][j];
    double v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = i0 + 8 * r;
      const double f = s[i][p] * ip;
      v[r] = i == p ? (j == p ? ip : pj * ip) : (j == p ? -f : fma(-f, pj, s[i][j]));
    }
    if (bj == k && threadIdx.x == 0 && !(piv > 0.0)) *bad = 1;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) s[i0 + 8 * r][j] = v[r];
    __syncthreads();
  }
  double v[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) v[r] = bj == k ? s[i0 + 8 * r][j] : 0.0;
  if (bj != k)
    for (int l = 0; l < kDiB; ++l)
#pragma unroll
      for (int r = 0; r < 4; ++r) v[r] = fma(s[i0 + 8 * r][l], X[l][j], v[r]);
#pragma unroll
  for (int r = 0; r < 4; ++r) R[(size_t)(i0 + 8 * r) * np + kDiB * bj + j] = v[r];
}

// B(k, j) = R(j); B(i, j) = A(i, j) - A(i, k) R(j), for j = k without the first term.
__global__ void __launch_bounds__(256) di_step_kernel(const double* __restrict__ A, double* __restrict__ B, int np,
                                                      int k, const double* __restrict__ R) {
  __shared__ double C[kDiB][kDiB + 1], X[kDiB][kDiB + 1];
  const int bi = blockIdx.y, bj = blockIdx.x, j = threadIdx.x & 31, i0 = threadIdx.x >> 5;
  double v[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int i = i0 + 8 * r;
    C[i][j] = A[(size_t)(kDiB * bi + i) * np + kDiB * k + j];
    X[i][j] = R[(size_t)i * np + kDiB * bj + j];
    v[r] = bi == k ? X[i][j] : (bj == k ? 0.0 : A[(size_t)(kDiB * bi + i) * np + kDiB * bj + j]);
  }
  __syncthreads();
  if (bi != k)
    for (int l = 0; l < kDiB; ++l)
#pragma unroll
      for (int r = 0; r < 4; ++r) v[r] = fma(-C[i0 + 8 * r][l], X[l][j], v[r]);
#pragma unroll
  for (int r = 0; r < 4; ++r) B[(size_t)(kDiB * bi + i0 + 8 * r) * np + kDiB * bj + j] = v[r];
}

// max |x| over the leading n x n, as the bits of a non-negative double (NaN: above all).
__global__ void __launch_bounds__(256) di_max_kernel(const double* __restrict__ A, int np, int n,
                                                     unsigned long long* __restrict__ out) {
  unsigned long long v = 0;
  for (int i = blockIdx.x; i < n; i += gridDim.x)
    for (int j = threadIdx.x; j < n; j += 256) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(A[(size_t)i * np + j]));
      v = b > v ? b : v;
    }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long b = __shfl_xor_sync(0xffffffffu, v, o);
    v = b > v ? b : v;
  }
  if ((threadIdx.x & 31) == 0) atomicMax(out, v);
}

// The fragments: 16 x 16 tile (mi, kk) at (mi nt + kk) 64 uint4, 32 lanes of heads and 32
// of tails; a lane's word q as in the factor's tiles.  Zero outside the n orbitals.
__global__ void __launch_bounds__(128) di_frag_kernel(const double* __restrict__ A, int np, int n, int nt, double sc,
                                                      uint32_t* __restrict__ fx) {
  const int mi = blockIdx.y, kk = blockIdx.x, l = threadIdx.x >> 2, q = threadIdx.x & 3;
  const int r = 16 * mi + (l >> 2) + 8 * (q & 1), k = 16 * kk + (l & 3) + 4 * (q >> 1);
  const float v0 = r < n && k < n ? (float)(A[(size_t)r * np + k] * sc) : 0.f;
  const float v1 = r < n && k + 8 < n ? (float)(A[(size_t)r * np + k + 8] * sc) : 0.f;
  uint32_t h, t;
  split_f16(v0, v1, h, t);
  uint32_t* f = fx + ((size_t)mi * nt + kk) * 256;
  f[l * 4 + q] = h;
  f[128 + l * 4 + q] = t;
}

}  // namespace gbk
