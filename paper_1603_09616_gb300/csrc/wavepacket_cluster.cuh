// Wavepacket propagation with a cluster of CS thread blocks per packet (the series and
// its terms: see the one-team kernel in solver.cu).
//
// A term's some 10^6 FP64 FMAs (1900 orbitals) run at two a clock on an SM, so one team
// per packet is bound by its own SM's FP64 pipe while most SMs have no packet.  Here
// the blocks of a cluster share them: each owns a contiguous range of the 64-row blocks
// in the H product, the triangular products and the updates, and RR = 64 / CS rows of
// every block in the two band chains.  The panel vectors stay in global memory, ordered
// by cluster barriers (five a term).
//
// The chain passes a block's 64 values on by st.async: each store completes bytes on an
// mbarrier of the receiving block, so a step costs one trip between SMs and no barrier.
// Two buffers are enough: nobody sends block i + 2 before it has block i + 1 whole, and
// every warp that sends block i + 1 has read block i.
//
// GB300, 32 packets of 1900 orbitals, 10 steps of 25 terms: 82.1 -> 27.5 ms with clusters
// of four (110 us a term; the FP64 FMAs of a quarter of a term are 58 us, the two chains'
// 60 hand-overs most of the rest).
#pragma once
#include "team_solver.cuh"

namespace gbk {

struct ClusterSmem {
  Smem sm;
  double2 y[2][64];
  unsigned long long bar[2];
  int fail;
};

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
// 8 bytes into the same place of cluster block `rank`, counted on its mbarrier.
__device__ __forceinline__ void send_f64(uint32_t dst, uint32_t bar, unsigned rank, double v) {
  uint32_t d, b;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(dst), "r"(rank));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(bar), "r"(rank));
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(d),
               "l"(__double_as_longlong(v)), "r"(b)
               : "memory");
}
// As mbar_wait_bounded, for data that other blocks of the cluster send.
__device__ __forceinline__ bool cluster_wait_bounded(unsigned long long* bar, uint32_t parity) {
  const unsigned long long t0 = global_ns();
  for (int it = 0; it < (1 << 20); ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((it & 15) == 15 && global_ns() - t0 > 200000000ull) break;
  }
  return false;
}

// y_i = t_i - E_i y_{i-1} (FWD) or x_i = u_i - F_i x_{i+1} for one column; four warps of
// every block of the cluster.  A thread is (row r of the block's RR, slice of k): slices
// are neighbouring lanes, whose partial sums meet by shuffles, real and imaginary parts
// on different lanes after the first.  The tile's values and t are loaded a step ahead.
// sends: blocks handed over before this pass.
template <int CS, bool FWD>
__device__ __noinline__ void cluster_chain(const Args& a, ClusterSmem& cs, const double2* t, double2* out,
                                           unsigned sends) {
  constexpr int RR = 64 / CS, NS = 128 / RR, LEN = 64 / NS;
  const int tid = threadIdx.x, s = tid % NS, row = (int)cluster_rank() * RR + tid / NS;
  const int N4 = 4 * a.m.nb, nblk = a.m.bf_nblk, bw = a.m.bf_bw, k0 = FWD ? 64 - bw : 0;
  const double* __restrict__ E = a.m.bf64 + (size_t)(FWD ? 2 : 3) * nblk * 4096 + (size_t)(k0 + s) * 64 + row;
  double e[LEN], tv = 0.0;
  auto load = [&](int st) {
    const int blk = FWD ? st : nblk - 1 - st;
#pragma unroll
    for (int i = 0; i < LEN; ++i)
      e[i] = st > 0 && st < nblk && s + NS * i < bw ? __ldg(E + (size_t)blk * 4096 + i * NS * 64) : 0.0;
    tv = s < 2 && st < nblk && 64 * blk + row < N4 ? reinterpret_cast<const double*>(t)[2 * (64 * blk + row) + s] : 0.0;
  };
  load(0);
  bool dead = cs.fail != 0;
  for (int st = 0; st < nblk; ++st) {
    const int blk = FWD ? st : nblk - 1 - st;
    double y = tv, ec[LEN];
#pragma unroll
    for (int i = 0; i < LEN; ++i) ec[i] = e[i];
    load(st + 1);
    if (st > 0) {
      const unsigned c = sends + st - 1;
      if (!dead && !cluster_wait_bounded(&cs.bar[c & 1], (c >> 1) & 1)) {
        cs.fail = 1;
        dead = true;
      }
      const double2* yb = cs.y[c & 1] + k0 + s;
      double2 acc = make_double2(0.0, 0.0);
#pragma unroll
      for (int i = 0; i < LEN; ++i) {
        if (NS * i >= bw) break;
        if (s + NS * i < bw) cfma(acc, ec[i], yb[NS * i]);
      }
      const double give = s & 1 ? acc.x : acc.y, keep = s & 1 ? acc.y : acc.x;
      double v = keep + __shfl_xor_sync(0xffffffffu, give, 1);
#pragma unroll
      for (int o = 2; o < NS; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      y -= v;
    }
    const unsigned c = sends + st;
    if (st + 1 < nblk) {
      if (tid == 0)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&cs.bar[c & 1])), "r"(1024)
                     : "memory");
      // the warp's reads of the buffer before last are over before any of its lanes sends
      __syncwarp();
      if (s < 2) {
        const uint32_t dst = smem_u32(&cs.y[c & 1][row]) + 8 * s, bar = smem_u32(&cs.bar[c & 1]);
        const double v = 64 * blk + row < N4 ? y : 0.0;
#pragma unroll
        for (int r = 0; r < CS; ++r) send_f64(dst, bar, r, v);
      }
    }
    if (s < 2 && 64 * blk + row < N4) reinterpret_cast<double*>(out)[2 * (64 * blk + row) + s] = y;
  }
}

template <int CS>
__global__ void __launch_bounds__(TPB, 1)
    wavepacket_cluster_kernel(const __grid_constant__ Args a, double2* __restrict__ psi, int nwp, int nsteps,
                              const double2* __restrict__ coef, int nterms, double ca, double cb, double2 phase,
                              char* __restrict__ scratch, size_t panel_bytes, int* __restrict__ status) {
  __shared__ ClusterSmem cs;
  const int rank = (int)cluster_rank(), p = blockIdx.x / CS, tid = threadIdx.x, n = a.m.n, nblk = a.m.bf_nblk;
  const int b0 = rank * nblk / CS, nb = (rank + 1) * nblk / CS - b0;           // own blocks
  const int r0 = 64 * b0, r1 = min(4 * a.m.nb, 64 * (b0 + nb));                // own rows
  char* base = scratch + (size_t)p * 7 * panel_bytes;
  auto panel = [&](int i) { return reinterpret_cast<double2*>(base + i * panel_bytes); };
  double2 *P = panel(0), *tm = panel(1), *tk = panel(2), *Y = panel(3), *HX = panel(4), *t1 = panel(5), *t2 = panel(6);
  if (tid < WMAX) cs.sm.act[tid] = tid == 0;
  if (tid == 0) {
    cs.fail = 0;
    mbar_init(&cs.bar[0], 1);
    mbar_init(&cs.bar[1], 1);
    fence_mbar_init();
  }
  for (int i = r0 + tid; i < r1; i += TPB) {
    P[i] = i < n ? psi[(size_t)i * nwp + p] : make_double2(0.0, 0.0);
    tm[i] = P[i];
  }
  cluster_sync();
  unsigned sends = 0;
  auto cm = [](double2 x, double2 y) { return make_double2(x.x * y.x - x.y * y.y, x.x * y.y + x.y * y.x); };
  // Y <- S^-1 H X on the own rows; X complete in the cluster.  The last pass ends without a
  // barrier: the caller's cluster barrier follows.
  auto apply_a = [&](const double2* X) {
    for (int i = r0 + tid; i < r1; i += TPB) HX[i] = row_d(a.m, a.m.hb, X, 1, 0, i);
    __syncthreads();
    bc_tri_f64<true, 1>(a, cs.sm, HX, t1, b0, nb);
    cluster_sync();
    if (tid < 128) cluster_chain<CS, true>(a, cs, t1, t1, sends);
    sends += nblk - 1;
    cluster_sync();
    bc_tri_f64<false, 1>(a, cs.sm, t1, t2, b0, nb);
    cluster_sync();
    if (tid < 128) cluster_chain<CS, false>(a, cs, t2, Y, sends);
    sends += nblk - 1;
    cluster_sync();
  };
  for (int step = 0; step < nsteps; ++step) {
    apply_a(tm);  // T_1 = (A T_0 - b T_0) / a; P <- c_0 T_0 + c_1 T_1
    for (int i = r0 + tid; i < r1; i += TPB) {
      const double2 t0 = tm[i];
      const double2 v = make_double2((Y[i].x - cb * t0.x) * ca, (Y[i].y - cb * t0.y) * ca);
      tk[i] = v;
      const double2 s0 = cm(coef[0], t0), s1 = cm(coef[1], v);
      P[i] = make_double2(s0.x + s1.x, s0.y + s1.y);
    }
    cluster_sync();
    for (int k = 2; k < nterms; ++k) {
      apply_a(tk);
      const double2 ck = coef[k];
      for (int i = r0 + tid; i < r1; i += TPB) {  // T_k = 2 (A T_{k-1} - b T_{k-1}) / a - T_{k-2}
        const double2 t1v = tk[i], t0v = tm[i];
        const double2 v = make_double2(2.0 * (Y[i].x - cb * t1v.x) * ca - t0v.x, 2.0 * (Y[i].y - cb * t1v.y) * ca - t0v.y);
        tm[i] = v;
        const double2 s = cm(ck, v);
        P[i] = make_double2(P[i].x + s.x, P[i].y + s.y);
      }
      cluster_sync();
      double2* sw = tm;
      tm = tk;
      tk = sw;
    }
    for (int i = r0 + tid; i < r1; i += TPB) {  // e^{-i b tau}; T_0 of the next step
      P[i] = cm(phase, P[i]);
      tm[i] = P[i];
    }
    cluster_sync();
  }
  for (int i = r0 + tid; i < min(r1, n); i += TPB) psi[(size_t)i * nwp + p] = P[i];
  if (tid == 0 && cs.fail) atomicOr(status, kStTimeout);
  cluster_sync();  // no block leaves while another may still send to it
}

}  // namespace gbk
