// The mixed path's factor solve on tensor cores: x = S^-1 f to FP32 accuracy.
//
// With the block factor of block_chol.cuh,
//   FWD  t_i = D_i^-1 f_i,   y_i = t_i - E_i y_{i-1}   (i ascending)
//   BWD  u_i = D_i^-T y_i,   x_i = u_i - F_i x_{i+1}   (i descending)
// the triangular products t, u of all blocks are independent: every warp of the
// team takes (block, 8 columns, half of the row tiles) tasks, its fragments read
// from L2 straight into registers (no other warp wants them).  Only the band
// products form a chain; one warp per 16 x 8 tile of a block walks it, its band
// tiles staged by TMA bulk copies two blocks ahead, the previous block's output
// handed over through shared memory, one barrier among the chain's warps per block.
//
// Arithmetic: m16n8k16 FP16 MMAs with FP32 accumulation on head / tail splits of
// both operands (22 bits; three products, tail x tail dropped).  The factor's
// fragments are split when the matrix is built (tile_kernel), the vector where it is
// produced or loaded, so the inner loop is loads and MMAs.  FP16's range is met by
// powers of two: the tiles' entries below 2^4, each column of f scaled to a maximum in
// (2^12, 2^13], and host-computed growth bounds that keep y and x below the scaled
// maximum of f.  Only factors that this range holds come here (factor_tiles).
//
// One solve is off by 3.4e-7 of the solution's largest entry (chains of 8 to 1900
// orbitals, mean over random and sparse right-hand sides; the TF32 passes 3.9e-7).  It
// is bound by the chain's latency, two steps a block.  GB300, one 512-thread team, cold
// caches, with the column maxima, against the TF32 passes (one step per block with both
// products, the splits in the inner loop, a 16-warp barrier): 16 real columns of 912
// orbitals 61 -> 44 us, of 1900 109 -> 70 us; 64 columns of 1900 260 -> 207 us.
#pragma once
#include <cuda_fp16.h>

namespace gbk {

__device__ __forceinline__ void split_f16(float x0, float x1, uint32_t& h, uint32_t& l) {
  const __half2 hh = __floats2half2_rn(x0, x1);
  const float2 f = __half22float2(hh);
  const __half2 ll = __floats2half2_rn(x0 - f.x, x1 - f.y);
  h = *reinterpret_cast<const uint32_t*>(&hh);
  l = *reinterpret_cast<const uint32_t*>(&ll);
}
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void named_sync(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Column maxima of a vector that a factor solve will take: this thread's column
// pair c = tid % W.  Every thread of the team calls it; a barrier must follow.
__device__ __forceinline__ void col_max(Smem& sm, int W, float m0, float m1) {
  for (int off = W; off < 32; off <<= 1) {
    m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, off));
    m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, off));
  }
  const int lane = threadIdx.x & 31;
  if (lane < W) {
    atomicMax(&sm.fmax[2 * lane], __float_as_uint(m0));
    atomicMax(&sm.fmax[2 * lane + 1], __float_as_uint(m1));
  }
}

__host__ __device__ inline int fx_block_words(int ne) { return (10 + 4 * ne) * 64; }  // uint4 per block and direction

// out = kd D^-1 (sc f) (FWD) or kd D^-T f (BWD) for every block.  `in`: element
// (row, col) at (row * R + col) * MUL (MUL = 2: the heads of a float-float vector).
template <bool FWD, int MUL>
__device__ __noinline__ void fx_tri(const Args& a, const Smem& sm, const float* __restrict__ in,
                                    float* __restrict__ out) {
  const int R = 2 * a.W, N4 = 4 * a.m.nb, nblk = a.m.bf_nblk, nt = R > 8 ? R / 8 : 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const float kd = a.m.fx_kd[FWD ? 0 : 1];
  const int bw4 = fx_block_words(a.m.fx_ne);
  for (int task = warp; task < 2 * nblk * nt; task += nwarp()) {
    const int half = task & 1, ni = (task >> 1) % nt, blk = (task >> 1) / nt;
    const uint4* __restrict__ A = a.m.fx + (size_t)(2 * blk + (FWD ? 0 : 1)) * bw4 + lane;
    const int col = 8 * ni + g;
    const bool cok = col < R;
    const float sc = FWD && cok ? sm.fsc[col] : 1.f;
    uint32_t bh[4][2], bl[4][2];
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      float v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {  // k pair t: rows t, t + 8; pair t + 4: rows t + 4, t + 12
        const int row = 64 * blk + 16 * kk + t + 8 * (q & 1) + 4 * (q >> 1);
        v[q] = cok && row < N4 ? in[((size_t)row * R + col) * MUL] : 0.f;
        if (FWD) v[q] *= sc;
      }
      split_f16(v[0], v[1], bh[kk][0], bl[kk][0]);
      split_f16(v[2], v[3], bh[kk][1], bl[kk][1]);
    }
    // half 0 and half 1 take five fragments each: the row tiles with 4 + 1 and 3 + 2 steps
#pragma unroll
    for (int part = 0; part < 2; ++part) {
      const int mi = half == 0 ? (part == 0 ? (FWD ? 3 : 0) : (FWD ? 0 : 3)) : (part == 0 ? (FWD ? 2 : 1) : (FWD ? 1 : 2));
      const int first = FWD ? mi * (mi + 1) / 2 : 4 * mi - mi * (mi - 1) / 2;
      float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        if (FWD ? kk > mi : kk < mi) continue;
        const uint4* f = A + (first + (FWD ? kk : kk - mi)) * 64;
        const uint4 ah = __ldg(f), al = __ldg(f + 32);
        mma_f16(d0, ah, bh[kk][0], bh[kk][1]);
        mma_f16(d1, ah, bl[kk][0], bl[kk][1]);
        mma_f16(d1, al, bh[kk][0], bh[kk][1]);
      }
      const int oc = 8 * ni + 2 * t;
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int row = 64 * blk + 16 * mi + g + 8 * hf;
        if (oc < R && row < N4)
          *reinterpret_cast<float2*>(out + (size_t)row * R + oc) =
              make_float2(kd * (d0[2 * hf] + d1[2 * hf]), kd * (d0[2 * hf + 1] + d1[2 * hf + 1]));
      }
    }
  }
}

// One thread: the band tile of chain step s (1 .. nblk - 1) into its stage.
template <bool FWD>
__device__ __forceinline__ void fx_issue(const Args& a, Smem& sm, unsigned base, int s) {
  extern __shared__ __align__(16) char bc_dyn[];
  const int ne = a.m.fx_ne, blk = FWD ? s : a.m.bf_nblk - 1 - s;
  const unsigned q = (base + (unsigned)s - 1u) % kTileBufs, stage = pass_layout(a.W, (a.bc_bw_alloc + 15) / 16).stage;
  fence_proxy_async_smem();
  tma_bulk_g2s(bc_dyn + q * stage, a.m.fx + (size_t)(2 * blk + (FWD ? 0 : 1)) * fx_block_words(ne) + 10 * 64,
               (uint32_t)ne * 4096u, &sm.bc_bar[q]);
}

// y_i = t_i - E_i y_{i-1} along the blocks, in place (FWD), or into x with the
// column's scale undone (BWD).  The first kTileBufs tiles are on their way.  A
// warp owns the 16 x 8 tile (mi, ni) of every block (NU = 2: also (mi, ni + 4)).
// One warp per scheduler is at work for 8 columns, so a step costs its dependent
// instructions: addresses advance by constants, the step is unrolled for NE band
// steps, and t is loaded two blocks ahead.  T and out may alias: a lane reads its t
// before it writes there.  The next tile is issued by the warp after the chain's
// (by the chain's first one if there is none): it took thread 0 455 of a step's 1340
// cycles.  Ends with a barrier of the team.
template <bool FWD, int NU, int NE>
__device__ __noinline__ void fx_chain(const Args& a, Smem& sm, const float* T, float* out) {
  extern __shared__ __align__(16) char bc_dyn[];
  const int R = 2 * a.W, N4 = 4 * a.m.nb, nblk = a.m.bf_nblk, nt = R > 8 ? R / 8 : 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int nw = 4 * nt / NU;  // warps of the chain
  const unsigned base = sm.tile_base;
  const bool spare = nw < nwarp();  // a warp to issue the tiles
  const int nsync = 32 * (nw + (spare ? 1 : 0));
  if (spare && warp == nw) {
    for (int s = 0; s < nblk; ++s) {
      named_sync(1, nsync);
      if (lane == 0 && s > 0 && s + kTileBufs < nblk) fx_issue<FWD>(a, sm, base, s + kTileBufs);
      __syncwarp();
    }
  } else if (warp < nw) {
    const PassLayout L = pass_layout(a.W, (a.bc_bw_alloc + 15) / 16);
    constexpr int P = kOutWords, k0 = FWD ? 4 - NE : 0, kp = k0 / 2, np = (k0 + NE + 1) / 2 - kp;  // pairs of band steps
    const int mi = warp & 3, ni = warp >> 2;
    uint32_t* ysm = reinterpret_cast<uint32_t*>(bc_dyn + L.o_y);
    // B fragments: lane l names row l % 8 of the 8 x 8 matrix l / 8 of a pair of band steps
    const uint32_t yr = smem_u32(ysm + (8 * ni + (lane & 7)) * P + 16 * kp + (lane >> 3) * 4);
    uint32_t* yw = ysm + (8 * ni + 2 * t) * P + 8 * mi + g;  // this lane's output words
    const int tails = (R > 8 ? R : 8) * P, buf = 2 * tails;
    const uint4* E0 = reinterpret_cast<const uint4*>(bc_dyn) + mi * NE * 64 + lane;
    const float ke = -a.m.fx_ke[FWD ? 0 : 1];
    const int first = FWD ? 0 : nblk - 1, row0 = 64 * first + 16 * mi + g, oc = 8 * ni + 2 * t;
    const ptrdiff_t dstep = (FWD ? 64 : -64) * (ptrdiff_t)R;
    const float* tp = T + (ptrdiff_t)row0 * R + oc;
    float* op = out + (ptrdiff_t)row0 * R + oc;
    bool ok[NU];
    float2 un[NU];
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      ok[u] = oc + 32 * u < R;
      un[u] = !FWD && ok[u] ? make_float2(sm.fun[oc + 32 * u], sm.fun[oc + 32 * u + 1]) : make_float2(1.f, 1.f);
    }
    // only the last block can be ragged: rows 64 i + 16 mi + g (+ 8) below N4
    const int last = nblk - 1;
    const bool r0 = 64 * last + 16 * mi + g < N4, r1 = 64 * last + 16 * mi + g + 8 < N4;
    const int ragged = FWD ? last : 0;
    unsigned q = base % kTileBufs, ph = (base / kTileBufs) & 1u;
    bool dead = sm.bc_fail != 0;
    auto load_t = [&](int s, float2 (&v)[NU][2]) {
      const bool in = s < nblk, g0 = in && (s != ragged || r0), g1 = in && (s != ragged || r1);
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        v[u][0] = ok[u] && g0 ? *reinterpret_cast<const float2*>(tp + 32 * u) : make_float2(0.f, 0.f);
        v[u][1] = ok[u] && g1 ? *reinterpret_cast<const float2*>(tp + 8 * R + 32 * u) : make_float2(0.f, 0.f);
      }
      tp += dstep;
    };
    auto step = [&](int s, float2 (&slot)[NU][2], uint32_t yprev, uint32_t* ynext) {
      float2 y[NU][2];
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        y[u][0] = slot[u][0];
        y[u][1] = slot[u][1];
      }
      load_t(s + 2, slot);
      if (s > 0) {
        if (!dead && !mbar_wait_bounded(&sm.bc_bar[q], ph)) {
          sm.bc_fail = 1;
          dead = true;
        }
        const uint4* E = E0 + q * (L.stage / 16);
#pragma unroll
        for (int u = 0; u < NU; ++u) {
          float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f}, d2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int pr = 0; pr < np; ++pr) {
            uint32_t h[4], l[4];
            ldmatrix4(h, yprev + (32 * u * P + 16 * pr) * 4);
            ldmatrix4(l, yprev + (32 * u * P + 16 * pr + tails) * 4);
#pragma unroll
            for (int o = 0; o < 2; ++o) {
              const int j = 2 * (kp + pr) + o - k0;
              if (j < 0 || j >= NE) continue;
              const uint4 ah = E[j * 64], al = E[j * 64 + 32];
              mma_f16(d0, ah, h[2 * o], h[2 * o + 1]);
              mma_f16(d1, ah, l[2 * o], l[2 * o + 1]);
              mma_f16(d2, al, h[2 * o], h[2 * o + 1]);
            }
          }
          y[u][0].x = fmaf(ke, d0[0] + (d1[0] + d2[0]), y[u][0].x);
          y[u][0].y = fmaf(ke, d0[1] + (d1[1] + d2[1]), y[u][0].y);
          y[u][1].x = fmaf(ke, d0[2] + (d1[2] + d2[2]), y[u][1].x);
          y[u][1].y = fmaf(ke, d0[3] + (d1[3] + d2[3]), y[u][1].y);
        }
        if (++q == kTileBufs) {
          q = 0;
          ph ^= 1u;
        }
      }
      // the block's output: FP16 words of row pairs (g, g + 8) for the next step
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        uint32_t h, l;
        uint32_t* w = ynext + 32 * u * P;
        split_f16(y[u][0].x, y[u][1].x, h, l);
        w[0] = h;
        w[tails] = l;
        split_f16(y[u][0].y, y[u][1].y, h, l);
        w[P] = h;
        w[P + tails] = l;
      }
      named_sync(1, nsync);
      const bool g0 = s != ragged || r0, g1 = s != ragged || r1;
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        if (ok[u] && g0) *reinterpret_cast<float2*>(op + 32 * u) = make_float2(y[u][0].x * un[u].x, y[u][0].y * un[u].y);
        if (ok[u] && g1)
          *reinterpret_cast<float2*>(op + 8 * R + 32 * u) = make_float2(y[u][1].x * un[u].x, y[u][1].y * un[u].y);
      }
      op += dstep;
      if (!spare && threadIdx.x == 0 && s > 0 && s + kTileBufs < nblk) fx_issue<FWD>(a, sm, base, s + kTileBufs);
    };
    float2 ta[NU][2], tb[NU][2];
    load_t(0, ta);
    load_t(1, tb);
    for (int s = 0; s < nblk; s += 2) {
      step(s, ta, yr + buf * 4, yw);
      if (s + 1 < nblk) step(s + 1, tb, yr, yw + buf);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) sm.tile_base = base + (unsigned)(nblk - 1);
}
template <bool FWD, int NU>
__device__ __forceinline__ void fx_chain_ne(const Args& a, Smem& sm, const float* T, float* out) {
  switch (a.m.fx_ne) {
    case 1: fx_chain<FWD, NU, 1>(a, sm, T, out); break;
    case 2: fx_chain<FWD, NU, 2>(a, sm, T, out); break;
    case 3: fx_chain<FWD, NU, 3>(a, sm, T, out); break;
    default: fx_chain<FWD, NU, 4>(a, sm, T, out); break;
  }
}

// x = S^-1 f for the panel's 2 W real columns (f: a float-float vector's heads,
// float4 pairs, or an FP32 vector, float2 pairs), every element finite or its
// column lost.  sm.fmax holds the column maxima of |f| (col_max; the barrier after
// it is passed); t1, t2: panel-sized scratch.  WIDE: W may exceed 16.  Ends with a
// barrier.
template <bool WIDE = false, typename InT>
__device__ void fx_solve(const Args& a, Smem& sm, const InT* f, float2* x, float2* t1, float2* t2) {
  constexpr int MUL = sizeof(InT) == 16 ? 2 : 1;
  const int tid = threadIdx.x;
  auto prologue = [&](auto fwd) {
    if (tid == 0) {
      const unsigned base = sm.tile_base;
      for (int s = 1; s <= kTileBufs && s < a.m.bf_nblk; ++s) fx_issue<decltype(fwd)::value>(a, sm, base, s);
    }
  };
  prologue(std::true_type{});
  if (tid < 2 * a.W) {
    const float m = __uint_as_float(sm.fmax[tid]);
    int ex = 0;
    if (m > 0.f && m < INFINITY) frexpf(m, &ex);
    const int k = m > 0.f ? max(-100, min(100, 13 - ex)) : 0;
    sm.fsc[tid] = ldexpf(1.f, k);
    sm.fun[tid] = ldexpf(1.f, max(-126, min(126, a.m.fx_lg - k)));
    sm.fmax[tid] = 0;
  }
  __syncthreads();
  float* y = reinterpret_cast<float*>(t1);
  float* u = reinterpret_cast<float*>(t2);
  fx_tri<true, MUL>(a, sm, reinterpret_cast<const float*>(f), y);
  __syncthreads();
  if (!WIDE || a.W <= 16)
    fx_chain_ne<true, 1>(a, sm, y, y);
  else if constexpr (WIDE)
    fx_chain_ne<true, 2>(a, sm, y, y);
  __syncthreads();  // tile_base
  prologue(std::false_type{});
  fx_tri<false, 1>(a, sm, y, u);
  __syncthreads();
  if (!WIDE || a.W <= 16)
    fx_chain_ne<false, 1>(a, sm, u, reinterpret_cast<float*>(x));
  else if constexpr (WIDE)
    fx_chain_ne<false, 2>(a, sm, u, reinterpret_cast<float*>(x));
  if (tid == 0) ++sm.inner_count;
  __syncthreads();
}

}  // namespace gbk
