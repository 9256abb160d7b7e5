// The factor solve of the seed recurrence's mixed path (panel.cuh): FWD and BWD
// passes with both products of a block in one step, on TF32 MMAs, whose operands keep
// an exponent per entry: they take every factor, also those outside FP16's range
// (factor_tiles), which gb_apply_sinv brings here too.  The others run the faster
// passes of factor_passes.cuh (its header has both times).
#pragma once

namespace gbk {

// ------------------------------------------------------------ FP32 passes on tensor cores
// One pass walks the blocks and forms, per block i (FWD, i ascending):
//   y_i = D_i^-1 f_i - E_i y_{i-1},
// (BWD, i descending: x_i = D_i^-T y_i - F_i x_{i+1}) as 64 x 2W products on
// m16n8k8 TF32 MMAs, one warp per 16 x 8 output tile.  FP32 accuracy from
// TF32 units: every operand is split into a TF32 head and a tail whose TF32
// part the units read (a = a_h + a_t to ~2^-21) and a b = a_h b_h + a_h b_t +
// a_t b_h is accumulated in FP32.  Per step: the block's tile (fragment order, built on
// the host) waits in its TMA stage, the input block was staged a step
// earlier, the previous output block sits in shared memory; one barrier.
// Head: x rounded to 11 significant bits (add half a TF32 unit to the bit
// pattern, clear the 13 low bits: exactly a TF32 value); tail: x - head,
// exact in FP32 and at most half a TF32 unit, of which the MMA reads the
// TF32 part (the units ignore the 13 low bits of a .tf32 operand).  Three
// full-rate integer / FP32 instructions per value.
__device__ __forceinline__ void split_tf32(float x, uint32_t& h, uint32_t& t) {
  h = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
  t = __float_as_uint(x - __uint_as_float(h));
}
__device__ __forceinline__ void mma_tf32(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// acc_h += A_h B_h, acc_t += A_h B_t + A_t B_h for one k-step: A fragment
// (four values of this lane) from the staged tile, B rows 8 ks + t, + 4 of
// column 8 ni + g of the block in shared memory (row stride P).
__device__ __forceinline__ void mma_kstep(float (&acc_h)[4], float (&acc_t)[4], float (&acc_u)[4],
                                          const float* __restrict__ frag, const float* __restrict__ B, int P, int ks,
                                          int ni, int lane) {
  const float4 av = *reinterpret_cast<const float4*>(frag + lane * 4);
  uint32_t ah[4], at[4];
  split_tf32(av.x, ah[0], at[0]);
  split_tf32(av.y, ah[1], at[1]);
  split_tf32(av.z, ah[2], at[2]);
  split_tf32(av.w, ah[3], at[3]);
  const int g = lane >> 2, t = lane & 3;
  uint32_t bh0, bt0, bh1, bt1;
  split_tf32(B[(8 * ks + t) * P + 8 * ni + g], bh0, bt0);
  split_tf32(B[(8 * ks + t + 4) * P + 8 * ni + g], bh1, bt1);
  mma_tf32(acc_h, ah, bh0, bh1);
  mma_tf32(acc_t, ah, bt0, bt1);
  mma_tf32(acc_u, at, bh0, bh1);
}
template <bool FWD, int PF, typename InT>
__device__ __noinline__ void bc_pass_mma(const Args& a, Smem& sm, const InT* __restrict__ in, float2* __restrict__ out) {
  const int W = a.W, N4 = 4 * a.m.nb, nblk = a.m.bf_nblk, bw = a.m.bf_bw, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const MmaLayout L = mma_layout(W, a.bc_bw_alloc);
  extern __shared__ __align__(16) char bc_dyn[];
  float* stage = reinterpret_cast<float*>(bc_dyn);
  float* fin = reinterpret_cast<float*>(bc_dyn + L.o_fin);
  float* ysm = reinterpret_cast<float*>(bc_dyn + L.o_ysm);
  float* xch = reinterpret_cast<float*>(bc_dyn + L.o_xch);
  const int P = L.P, S = L.S, ntile = 4 * L.nt;
  const int ksE0 = (64 - bw) / 8, nF = (bw + 7) / 8;
  const int n2 = FWD ? 8 - ksE0 : nF;  // band k-steps
  const uint32_t tile_bytes = (uint32_t)(20 + 4 * n2) * 512u;
  const float* tiles = a.m.bfm + (FWD ? 0 : kMmaTileFloatsDev);
  const unsigned base = sm.tile_base;
  auto blk_of = [&](int s) { return FWD ? s : nblk - 1 - s; };
  auto issue = [&](int s) {  // thread 0: the tile of step s into stage (base + s) % S
    const unsigned q = base + (unsigned)s;
    fence_proxy_async_smem();
    tma_bulk_g2s(stage + (q % S) * L.stage_floats, tiles + (size_t)(2 * blk_of(s)) * kMmaTileFloatsDev, tile_bytes,
                 &sm.bc_bar[q % S]);
  };
  // input blocks: this thread's PF complex values of a block, DEPTH blocks ahead
  constexpr int DEPTH = PF == 1 ? 3 : 2;
  float2 pq[DEPTH][PF];
  auto load_block = [&](float2 (&dst)[PF], int s) {
    const int i = blk_of(s);
#pragma unroll
    for (int m = 0; m < PF; ++m) {
      const int o = tid + m * TPB;
      const int row = 64 * i + o / W;
      dst[m] = (s < nblk && o < 64 * W && row < N4) ? bc_in(in, (size_t)64 * i * W + o) : make_float2(0.f, 0.f);
    }
  };
  auto store_block = [&](const float2 (&src)[PF], float* dst) {
#pragma unroll
    for (int m = 0; m < PF; ++m) {
      const int o = tid + m * TPB;
      if (o < 64 * W) {
        const int r = o / W, c = o - r * W;
        *reinterpret_cast<float2*>(dst + r * P + 2 * c) = src[m];
      }
    }
  };
  // prologue: zero both staging areas (padding columns stay zero), stage
  // block 0, queue blocks 1..DEPTH, issue the first tiles
  for (int e = tid; e < 4 * 64 * P; e += TPB) fin[e] = 0.f;  // fin and ysm are adjacent
  if (tid == 0)
    for (int s = 0; s < S - 1 && s < nblk; ++s) issue(s);
  {
    float2 b0[PF];
    load_block(b0, 0);
#pragma unroll
    for (int d = 0; d < DEPTH; ++d) load_block(pq[(1 + d) % DEPTH], 1 + d);
    __syncthreads();  // zeroing done before the stores below
    store_block(b0, fin);
  }
  __syncthreads();
  // One step per block.  The register queue of input blocks rotates by slot
  // (the loop is unrolled DEPTH times so the slots stay registers): step s
  // stages block s + 1 from slot (s + 1) % DEPTH and refills that slot with
  // block s + 1 + DEPTH.
  auto step = [&](int s, float2 (&slot)[PF]) {
    const int i = blk_of(s);
    const float* fcur = fin + (s & 1) * 64 * P;
    const float* yprev = ysm + ((s + 1) & 1) * 64 * P;
    float* ycur = ysm + (s & 1) * 64 * P;
    if (s + 1 < nblk) {  // stage the next input block (its buffer was read a step ago)
      store_block(slot, fin + ((s + 1) & 1) * 64 * P);
      load_block(slot, s + 1 + DEPTH);
    }
    if (tid == 0 && s + S - 1 < nblk) issue(s + S - 1);
    const unsigned q = base + (unsigned)s;
    if (!sm.bc_fail && !mbar_wait_bounded(&sm.bc_bar[q % S], (q / S) & 1u)) sm.bc_fail = 1;
    const float* T = stage + (q % S) * L.stage_floats;
    // Up to eight tiles (W <= 8): warp w < ntile forms the triangular part of
    // tile w, warp ntile + w its band part, and hands it over through shared
    // memory (a named barrier per pair); more tiles: one warp per tile.
    const bool split = 2 * ntile <= NWARP;
    const int nunits = split ? 2 * ntile : ntile;
    for (int u = warp; u < nunits; u += NWARP) {
      const int ot = split ? u % ntile : u, role = split ? u / ntile : 2;  // 0 tri, 1 band, 2 both
      // Warp w runs on sub-partition w mod 4.  The triangular part of m-tile
      // mi takes 2 mi + 2 (FWD) or 8 - 2 mi (BWD) k-steps, so odd n-tiles run
      // the m-tiles in reverse: every sub-partition then issues the same
      // number of tensor instructions per step (10 k-steps of triangle per
      // pair of n-tiles instead of 4 .. 16).
      const int ni = ot >> 2, mi = (ni & 1) ? 3 - (ot & 3) : (ot & 3);
      float dh[4] = {0.f, 0.f, 0.f, 0.f}, dt[4] = {0.f, 0.f, 0.f, 0.f}, du[4] = {0.f, 0.f, 0.f, 0.f};
      float e[4] = {0.f, 0.f, 0.f, 0.f};
      if (role != 0 && s > 0) {  // band part against the previous output block
        const int kb = FWD ? ksE0 : 0;
        for (int j = 0; j < n2; ++j) mma_kstep(dh, dt, du, T + (20 + 4 * j + mi) * 128, yprev, P, kb + j, ni, lane);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          e[v] = dh[v] + (dt[v] + du[v]);
          dh[v] = dt[v] = du[v] = 0.f;
        }
      }
      if (role == 1) {
        *reinterpret_cast<float4*>(xch + (ot * 32 + lane) * 4) = make_float4(e[0], e[1], e[2], e[3]);
        named_sync(1 + ot, 64);
        continue;
      }
      // triangular part: FWD lower (k-steps 0 .. 2 mi + 1), BWD upper (2 mi .. 7)
      const int k0 = FWD ? 0 : 2 * mi, k1 = FWD ? 2 * mi + 2 : 8;
      for (int ks = k0; ks < k1; ++ks) {
        // fragment index: FWD pairs (ks, mi >= ks / 2) after sum_{s < ks} (4 - s / 2);
        // BWD pairs (ks, mi <= ks / 2) after sum_{s < ks} (s / 2 + 1)
        const int h = ks >> 1;
        const int pre = FWD ? 4 * ks - (h * (h - 1) + (ks & 1) * h) : (h * (h + 1) + (ks & 1) * (h + 1));
        const int pair = FWD ? pre + mi - h : pre + mi;
        mma_kstep(dh, dt, du, T + pair * 128, fcur, P, ks, ni, lane);
      }
      if (role == 0) {
        named_sync(1 + ot, 64);
        const float4 ev = *reinterpret_cast<const float4*>(xch + (ot * 32 + lane) * 4);
        e[0] = ev.x;
        e[1] = ev.y;
        e[2] = ev.z;
        e[3] = ev.w;
      }
      const int cc = 4 * ni + t;  // complex column of this lane's outputs
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int r = 16 * mi + g + 8 * hf, row = 64 * i + r;
        float2 y = make_float2((dh[2 * hf] + (dt[2 * hf] + du[2 * hf])) - e[2 * hf],
                               (dh[2 * hf + 1] + (dt[2 * hf + 1] + du[2 * hf + 1])) - e[2 * hf + 1]);
        if (row >= N4) y = make_float2(0.f, 0.f);
        *reinterpret_cast<float2*>(ycur + r * P + 8 * ni + 2 * t) = y;
        if (cc < W && row < N4 && sm.act[cc]) out[(size_t)row * W + cc] = y;
      }
    }
    if (tid == 0 && s + 1 == nblk) sm.tile_base = base + (unsigned)nblk;  // every thread read it at entry
    __syncthreads();
  };
  for (int s0 = 0; s0 < nblk; s0 += DEPTH) {
#pragma unroll
    for (int j = 0; j < DEPTH; ++j)
      if (s0 + j < nblk) step(s0 + j, pq[(j + 1) % DEPTH]);
  }
}

// x = S^-1 f for every active column; t1: panel-sized scratch.  Ends with a barrier.
template <int PF, typename InT>
__device__ void seed_solve_w(const Args& a, Smem& sm, const InT* f, float2* x, float2* t1) {
  bc_pass_mma<true, PF>(a, sm, f, t1);
  bc_pass_mma<false, PF>(a, sm, t1, x);
  if (threadIdx.x == 0) ++sm.inner_count;
}
template <typename InT>
__device__ void seed_solve(const Args& a, Smem& sm, const InT* f, float2* x, float2* t1) {
  if (a.W == 32)
    seed_solve_w<4>(a, sm, f, x, t1);
  else if (a.W == 16)
    seed_solve_w<2>(a, sm, f, x, t1);
  else
    seed_solve_w<1>(a, sm, f, x, t1);
}

}  // namespace gbk
