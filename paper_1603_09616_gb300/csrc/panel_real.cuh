// The real three-term recurrence: the panel solver of every solve that does
// not ask for the seed recurrence (panel.cuh).
//
// b = e_j, H and S are real, so the Krylov space of A = S^-1 H and b that every
// shift shares has a real basis, whatever the shifts are.  The basis is built by
// the three-term recurrence in the S inner product, with s_n = S v_n carried
// beside v_n and neither normalised (s_0 = e_j, b_n^2 = s_n^T v_n):
//   v_n = S^-1 s_n,  U = H v_n,  a_n = v_n^T U / b_n^2,
//   s_{n+1} = c1 U - c2 s_n - c3 s_{n-1},   c1 = 1 / b_n, c2 = a_n / b_n, c3 = b_n / b_{n-1}.
// So s_n = P_n(H S^-1) e_j, and the Galerkin solution of shift z in the space
// of dimension n has the residual s_n / P_n(z), P_n from the same recurrence:
//   P_{n+1} = (c1 z - c2) P_n - c3 P_{n-1},   P_0 = 1, P_{-1} = 0.
// It is the iterate of shifted COCG, without its seed: no coefficient depends
// on a shift, none can break down (b_n > 0 for an SPD S until the space is
// exhausted), and every vector keeps a norm of order b_n.  The solution is
//   x = sum_m y_m v_m,  y_m = (P_m / b_m^2) Q_m,  Q_m = sum_{l = m}^{n-1} b_l / (P_l P_{l+1}),
// whose sum runs backward over the recorded scalars, replayed from checkpoints.
//
// Two real columns take the place of one complex column: a panel of W pairs
// uses the vectors, sparse products and factor solves of a complex panel of
// width W for 2 W right-hand sides, which is what halves the cost of an
// iteration; the updates and dots shrink more (no complex arithmetic, 3 vectors
// instead of 6).
#pragma once
#include "panel.cuh"

namespace gbk {

constexpr int RMAX = 32;  // right-hand sides per panel

struct RealSmem : Smem {
  int j[RMAX], mc[RMAX], off[RMAX + 1], on[RMAX], nc[RMAX], nact[RMAX], nfresh[RMAX], cst[RMAX];
  double b2[RMAX], c1prev[RMAX], c1[RMAX], c2[RMAX], c3[RMAX], s2[RMAX];
  float2 f1[RMAX], f2[RMAX], f3[RMAX];  // c1, -c2, -c3 as float-floats
  int Mt[RMAX * 8];  // replay length per (column, 32-shift group)
  int Mc[RMAX];
};

// The next value of the shift polynomial; explicit roundings, so that the loop
// and the replay form identical values.
__device__ __forceinline__ double2 real_step(double2 cur, double2 prev, double c1, double c2, double c3, double2 z) {
  const double zr = fma(c1, z.x, -c2), zi = __dmul_rn(c1, z.y);
  return make_double2(fma(zr, cur.x, fma(-zi, cur.y, -__dmul_rn(c3, prev.x))),
                      fma(zr, cur.y, fma(zi, cur.x, -__dmul_rn(c3, prev.y))));
}

// Both real columns of a stored pair, as FP64.
__device__ __forceinline__ double pair_part(double2 v, int p) { return p ? v.y : v.x; }
__device__ __forceinline__ double pair_part(float4 v, int p) {
  return p ? (double)v.z + (double)v.w : (double)v.x + (double)v.y;
}

// v_m on the pattern rows of every column of the panel -> one history row.
template <bool MIX>
__device__ void gather_real(const Args& a, const RealSmem& sm, const SeedT<MIX>* v, double* row) {
  const int R = 2 * a.W;
  if (a.full_hist) {  // every row of every column: row[cc * N4 + i]
    const int N4 = 4 * a.m.nb;
    for (int e = threadIdx.x; e < N4 * R; e += tpb()) {
      const int cc = e / N4, i = e - cc * N4;
      row[e] = pair_part(v[(size_t)i * a.W + (cc >> 1)], cc & 1);
    }
    return;
  }
  const int M = sm.off[R];
  for (int e = threadIdx.x; e < M; e += tpb()) {
    int cc = 0;
    while (sm.off[cc + 1] <= e) ++cc;
    const int i = a.m.col_idx[a.m.row_ptr[sm.j[cc]] + e - sm.off[cc]];
    row[e] = pair_part(v[(size_t)i * a.W + (cc >> 1)], cc & 1);
  }
}

template <bool MIX>
__device__ void solve_panel_real(const Args& a, RealSmem& sm, char* ws, char* dyn) {
  using V = SeedT<MIX>;
  const int W = a.W, R = 2 * W, K = a.K, tid = threadIdx.x, c = tid % W;
  const size_t NE = (size_t)4 * a.m.nb * W;
  V* s = wsp<V>(ws, a.o_r);    // s_n
  V* so = wsp<V>(ws, a.o_rt);  // s_{n-1}, then s_{n+1}
  V* v = wsp<V>(ws, a.o_w);
  V* U = wsp<V>(ws, a.o_u);
  double* hr = wsp<double>(ws, a.o_hr);
  double* hc = wsp<double>(ws, a.o_ab);  // c1, c2, c3 per (iteration, column)
  double* ht = wsp<double>(ws, a.o_t);   // (S v_m)_j = s_m[j]
  double2* ck = wsp<double2>(ws, a.o_ck);
  double2* pis = wsp<double2>(ws, a.o_pi);
  int* nk = wsp<int>(ws, a.o_nk);
  double* resk = wsp<double>(ws, a.o_res);
  double2* buf = wsp<double2>(ws, a.o_buf);
  double* cp = wsp<double>(ws, a.o_cp);
  double* cf = wsp<double>(ws, a.o_cf);
  double2* cgs = a.want_g ? wsp<double2>(ws, a.o_cg) : nullptr;
  const int RK = R * K;
  using CgT = typename std::conditional<MIX, float2, double2>::type;
  CgT* cg_x = wsp<CgT>(ws, a.o_x);
  CgT* cg_g = a.cg_smem ? reinterpret_cast<CgT*>(dyn + dyn_layout(!MIX, W, false, 0).o_cg) : wsp<CgT>(ws, a.o_g);
  CgT* cg_d = a.cg_smem ? cg_g + NE : wsp<CgT>(ws, a.o_d);
  CgT* cg_q = a.cg_smem ? cg_d + NE : wsp<CgT>(ws, a.o_q);

  // ---------------------------------------------------------------- set-up
  if (tid < RMAX) {
    const int col = sm.panel * a.C + tid;
    const bool ok = tid < a.C && col < a.nrhs;
    const int jj = ok ? a.rhs_cols[col] : 0;
    sm.j[tid] = jj;
    sm.on[tid] = ok ? 1 : 0;
    sm.mc[tid] = ok ? a.m.row_ptr[jj + 1] - a.m.row_ptr[jj] : 0;
    sm.nc[tid] = 0;
    sm.cst[tid] = 0;
    sm.nact[tid] = 0;
    sm.nfresh[tid] = 0;
    sm.c1prev[tid] = 0.0;
    sm.c1[tid] = sm.c2[tid] = sm.c3[tid] = 0.0;
    sm.s2[tid] = 1.0;
  }
  if (tid < WMAX) sm.st[tid] = 0;
  __syncthreads();
  if (tid == 0) {
    sm.off[0] = 0;
    for (int i = 0; i < R; ++i) sm.off[i + 1] = sm.off[i] + sm.mc[i];
    sm.inner_count = 0;
  }
  if (tid < W) sm.act[tid] = sm.on[2 * tid] | sm.on[2 * tid + 1];
  for (int e = tid; e < RK; e += tpb()) {
    nk[e] = sm.on[e / K] ? -1 : 0;
    resk[e] = 0.0;
    pis[2 * e] = make_double2(1.0, 0.0);
    pis[2 * e + 1] = make_double2(0.0, 0.0);
    ck[2 * e] = make_double2(1.0, 0.0);
    ck[2 * e + 1] = make_double2(0.0, 0.0);
  }
  for (size_t e = tid; e < NE; e += tpb()) {
    const int row = (int)(e / W);
    const double x = sm.on[2 * c] && row == sm.j[2 * c] ? 1.0 : 0.0;
    const double y = sm.on[2 * c + 1] && row == sm.j[2 * c + 1] ? 1.0 : 0.0;
    if constexpr (MIX) {
      s[e] = make_float4((float)x, 0.f, (float)y, 0.f);
      so[e] = make_float4(0.f, 0.f, 0.f, 0.f);
      v[e] = make_float4(0.f, 0.f, 0.f, 0.f);
      U[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
      s[e] = make_double2(x, y);
      so[e] = v[e] = U[e] = make_double2(0.0, 0.0);
    }
  }
  __syncthreads();

  // v = S^-1 f and b2 = f^T v for the active pairs
  auto apply_sinv = [&](const V* f) {
    double d[2] = {0, 0};
    if constexpr (MIX) {
      gbff::acc d0, d1;
      gbff::acc_init(d0);
      gbff::acc_init(d1);
      const int e0 = sm.act[c] ? tid : (int)NE;
      const bool factor = a.inner_bchol || a.inner_dense;
      int levels = 0;
      if (factor)
        levels = inner_real_factor(a, sm, f, cg_x, cg_g, cg_d, cg_q, U);
      else
        inner_mixed<true>(a, sm, f, v, cg_x, cg_g, cg_d, cg_q, dyn);
      const float2 *x0 = cg_x, *x1 = cg_x + NE, *x2 = cg_g + NE, *x3 = cg_d + NE;
#pragma unroll 2
      for (int e = e0; e < (int)NE; e += tpb()) {
        const float4 fv = f[e];
        float4 vv;
        if (factor) {  // v = the levels' sum, smallest first
          gbff::ff p{0.f, 0.f}, q{0.f, 0.f};
          if (levels > 3) {
            const float2 t = x3[e];
            p.hi = t.x;
            q.hi = t.y;
          }
          if (levels > 2) {
            const float2 t = x2[e];
            p = gbff::two_sum(t.x, p.hi);
            q = gbff::two_sum(t.y, q.hi);
          }
          if (levels > 1) {
            const float2 t = x1[e];
            p = gbff::ff_add(gbff::ff{t.x, 0.f}, p);
            q = gbff::ff_add(gbff::ff{t.y, 0.f}, q);
          }
          const float2 t = x0[e];
          p = gbff::ff_add(gbff::ff{t.x, 0.f}, p);
          q = gbff::ff_add(gbff::ff{t.y, 0.f}, q);
          vv = make_float4(p.hi, p.lo, q.hi, q.lo);
          v[e] = vv;
        } else {
          vv = v[e];
        }
        gbff::acc_mul_add(d0, gbff::ff{fv.x, fv.y}, gbff::ff{vv.x, vv.y});
        gbff::acc_mul_add(d1, gbff::ff{fv.z, fv.w}, gbff::ff{vv.z, vv.w});
      }
      block_reduce_acc(d0, d1, W, sm.rs);
    } else {
      inner64(a, sm, f, v, cg_g, cg_d, cg_q, dyn);
#pragma unroll 4
      for (size_t e = sm.act[c] ? tid : NE; e < NE; e += tpb()) {
        const V fv = f[e], vv = v[e];
        d[0] = fma(fv.x, vv.x, d[0]);
        d[1] = fma(fv.y, vv.y, d[1]);
      }
      block_reduce_tree<2>(d, W, sm.rs);
    }
    if (tid < R) sm.b2[tid] = sm.rs.scal[(tid & 1) * WMAX + (tid >> 1)];
    __syncthreads();
  };
  if (tid < R) sm.fmax[tid] = __float_as_uint(1.f);
  __syncthreads();
  apply_sinv(s);
  gather_real<MIX>(a, sm, v, hr);
  if (tid < R) ht[tid] = 1.0;  // s_0[j]

  // ---------------------------------------------------------------- recurrence
  const double tol2 = a.tol * a.tol;
  int n = 0;
  for (; n < a.maxit; ++n) {
    if (tid == 0) {
      int any = 0;
      for (int i = 0; i < W; ++i) any |= sm.act[i];
      sm.flag = any;
    }
    __syncthreads();
    if (!sm.flag) break;

    {  // U = H v, v^T U
      double d[2] = {0, 0};
      gbff::acc d0, d1;
      gbff::acc_init(d0);
      gbff::acc_init(d1);
      for (int e = tid; e < (int)NE; e += tpb()) {
        if (!sm.act[c]) continue;
        const int row = e / W;
        if constexpr (MIX) {
          gbff::acc x0, x1;
          if (a.hp_fp32) {  // unrefined FP32 product: U = H hi(v), accumulated in FP32
            const float2 u = row_f(a.m, a.m.hb_hi, v, W, c, row);
            x0 = gbff::acc{u.x, 0.f};
            x1 = gbff::acc{u.y, 0.f};
          } else {
            row_ff(a.m, a.m.hb_hi, a.m.hb_lo, v, W, c, row, x0, x1);
          }
          const gbff::ff u0 = gbff::acc_get(x0), u1 = gbff::acc_get(x1);
          const float4 vv = v[e];
          U[e] = make_float4(u0.hi, u0.lo, u1.hi, u1.lo);
          gbff::acc_mul_add(d0, gbff::ff{vv.x, vv.y}, u0);
          gbff::acc_mul_add(d1, gbff::ff{vv.z, vv.w}, u1);
        } else {
          const double2 u = row_d(a.m, a.m.hb, v, W, c, row), vv = v[e];
          U[e] = u;
          d[0] = fma(vv.x, u.x, d[0]);
          d[1] = fma(vv.y, u.y, d[1]);
        }
      }
      if constexpr (MIX)
        block_reduce_acc(d0, d1, W, sm.rs);
      else
        block_reduce_tree<2>(d, W, sm.rs);
      if (tid < R) {
        double c1 = 0.0, c2 = 0.0, c3 = 0.0;
        if (sm.on[tid]) {
          const double b2 = sm.b2[tid];
          c1 = rsqrt(b2);
          c2 = sm.rs.scal[(tid & 1) * WMAX + (tid >> 1)] * (c1 * c1) * c1;
          c3 = b2 * c1 * sm.c1prev[tid];
          if (!(b2 > 0.0) || !isfinite(c1) || !isfinite(c2) || !isfinite(c3)) {
            // s^T S^-1 s <= 0 for a nonzero s: S is not positive definite
            sm.cst[tid] |= b2 < 0.0 ? kStNotSPD : kStBreakdown;
            sm.on[tid] = 0;
            sm.nc[tid] = n;
            c1 = c2 = c3 = 0.0;
          } else {
            sm.c1prev[tid] = c1;
            double* h = hc + ((size_t)n * R + tid) * 3;
            h[0] = c1;
            h[1] = c2;
            h[2] = c3;
          }
        }
        sm.c1[tid] = c1;
        sm.c2[tid] = c2;
        sm.c3[tid] = c3;
        if constexpr (MIX) {
          const gbff::ff g1 = gbff::ff_from_double(c1), g2 = gbff::ff_from_double(-c2), g3 = gbff::ff_from_double(-c3);
          sm.f1[tid] = make_float2(g1.hi, g1.lo);
          sm.f2[tid] = make_float2(g2.hi, g2.lo);
          sm.f3[tid] = make_float2(g3.hi, g3.lo);
        }
        sm.nact[tid] = 0;
        sm.nfresh[tid] = 0;
      }
      __syncthreads();
    }

    {  // s_{n+1} = c1 U - c2 s_n - c3 s_{n-1} (zero for a finished column), ||s_{n+1}||^2
      double d[2] = {0, 0};
      gbff::acc d0, d1;
      gbff::acc_init(d0);
      gbff::acc_init(d1);
      float m0 = 0.f, m1 = 0.f;  // max |s|, for the factor solve's scale
      if constexpr (MIX) {
        const gbff::ff fp0{sm.f1[2 * c].x, sm.f1[2 * c].y}, fp1{sm.f1[2 * c + 1].x, sm.f1[2 * c + 1].y};
        const gbff::ff fq0{sm.f2[2 * c].x, sm.f2[2 * c].y}, fq1{sm.f2[2 * c + 1].x, sm.f2[2 * c + 1].y};
        const gbff::ff ft0{sm.f3[2 * c].x, sm.f3[2 * c].y}, ft1{sm.f3[2 * c + 1].x, sm.f3[2 * c + 1].y};
#pragma unroll 2
        for (size_t e = sm.act[c] ? tid : NE; e < NE; e += tpb()) {
          const float4 u = U[e], x = s[e], y = so[e];
          const gbff::ff r0 = gbff::ff_add(gbff::ff_mul(fp0, gbff::ff{u.x, u.y}),
                                           gbff::ff_add(gbff::ff_mul(fq0, gbff::ff{x.x, x.y}),
                                                        gbff::ff_mul(ft0, gbff::ff{y.x, y.y})));
          const gbff::ff r1 = gbff::ff_add(gbff::ff_mul(fp1, gbff::ff{u.z, u.w}),
                                           gbff::ff_add(gbff::ff_mul(fq1, gbff::ff{x.z, x.w}),
                                                        gbff::ff_mul(ft1, gbff::ff{y.z, y.w})));
          so[e] = make_float4(r0.hi, r0.lo, r1.hi, r1.lo);
          m0 = fmaxf(m0, fabsf(r0.hi));
          m1 = fmaxf(m1, fabsf(r1.hi));
          gbff::acc_mul_add(d0, r0, r0);
          gbff::acc_mul_add(d1, r1, r1);
        }
        col_max(sm, W, m0, m1);
      } else {
        const double p0 = sm.c1[2 * c], p1 = sm.c1[2 * c + 1], q0 = sm.c2[2 * c], q1 = sm.c2[2 * c + 1];
        const double t0 = sm.c3[2 * c], t1 = sm.c3[2 * c + 1];
#pragma unroll 2
        for (size_t e = sm.act[c] ? tid : NE; e < NE; e += tpb()) {
          const double2 u = U[e], x = s[e], y = so[e];
          const double r0 = fma(p0, u.x, fma(-q0, x.x, -t0 * y.x)), r1 = fma(p1, u.y, fma(-q1, x.y, -t1 * y.y));
          so[e] = make_double2(r0, r1);
          d[0] = fma(r0, r0, d[0]);
          d[1] = fma(r1, r1, d[1]);
        }
      }
      if constexpr (MIX)
        block_reduce_acc(d0, d1, W, sm.rs);
      else
        block_reduce_tree<2>(d, W, sm.rs);
      if (tid < R && sm.on[tid]) {
        const double s2 = sm.rs.scal[(tid & 1) * WMAX + (tid >> 1)];
        if (isfinite(s2)) {
          sm.s2[tid] = s2;
        } else {
          sm.cst[tid] |= kStBreakdown;
          sm.on[tid] = 0;
          sm.nc[tid] = n;
        }
      }
      __syncthreads();
      V* w = s;  // s_{n+1} becomes the current vector
      s = so;
      so = w;
    }

    // shift polynomials, convergence, checkpoints
    for (int e = tid; e < RK; e += tpb()) {
      const int cc = e / K;
      if (!sm.on[cc] || nk[e] >= 0) continue;
      const double2 cur = pis[2 * e], nxt = real_step(cur, pis[2 * e + 1], sm.c1[cc], sm.c2[cc], sm.c3[cc], a.z[e - cc * K]);
      const double p2 = cabs2(nxt);
      if (sm.s2[cc] <= tol2 * p2) {
        nk[e] = n + 1;
        resk[e] = sqrt(sm.s2[cc] / p2);
      } else {
        atomicAdd(&sm.nact[cc], 1);
        if (a.stall > 0) {
          // while the pair is open, resk holds its best squared residual so far
          // and nk = -2 - (iteration of that best); both are rewritten when the
          // column ends
          const double r2 = sm.s2[cc] / p2, best = resk[e];
          if (nk[e] == -1 || r2 < 0.25 * best) {
            resk[e] = r2;
            nk[e] = -2 - n;
          }
          if (n - (-2 - nk[e]) < a.stall) atomicAdd(&sm.nfresh[cc], 1);
        }
      }
      pis[2 * e] = nxt;
      pis[2 * e + 1] = cur;
      if ((n + 1) % CK == 0) {
        const size_t ce = ((size_t)((n + 1) / CK) * RK + e) * 2;
        ck[ce] = nxt;
        ck[ce + 1] = cur;
      }
    }
    if (tid < R && sm.on[tid])
      ht[(size_t)(n + 1) * R + tid] = pair_part(s[(size_t)sm.j[tid] * W + (tid >> 1)], tid & 1);
    apply_sinv(s);  // its barriers order the counts above
    gather_real<MIX>(a, sm, v, hr + (size_t)(n + 1) * a.Mcap);
    if (tid < R && sm.on[tid]) {
      if (sm.nact[tid] == 0) {
        sm.on[tid] = 0;
        sm.nc[tid] = n + 1;
      } else if (a.stall > 0 && sm.nfresh[tid] == 0) {  // every open shift has stalled
        sm.on[tid] = 0;
        sm.nc[tid] = n + 1;
        sm.cst[tid] |= kStNoConv | kStStall;
      }
    }
    __syncthreads();
    if (tid < W) sm.act[tid] = sm.on[2 * tid] | sm.on[2 * tid + 1];
    __syncthreads();
  }
  if (tid < R && sm.on[tid]) {  // iteration cap reached
    sm.on[tid] = 0;
    sm.nc[tid] = n;
    sm.cst[tid] |= kStNoConv;
  }
  __syncthreads();
  for (int e = tid; e < RK; e += tpb()) {
    const int cc = e / K;
    if (sm.mc[cc] != 0 && nk[e] < 0) {
      nk[e] = sm.nc[cc];
      resk[e] = sqrt(sm.s2[cc] / cabs2(pis[2 * e]));
    }
  }
  __syncthreads();

  // ---------------------------------------------------------------- final phase
  const int KG = a.KG;
  // F1: backward sums per (column, 32 shifts), the polynomials replayed from checkpoints
  {
    const int lane = tid & 31, warp = tid >> 5;
    for (int task = warp; task < R * KG; task += nwarp()) {
      const int cc = task / KG, kg = task - cc * KG;
      if (sm.mc[cc] == 0) {
        if (lane == 0) sm.Mt[task] = 0;
        continue;
      }
      const int k = kg * 32 + lane;
      const bool valid = k < K;
      const int e = cc * K + (valid ? k : 0);
      const int nkk = valid ? nk[e] : 0;
      int M = nkk;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) M = max(M, __shfl_xor_sync(0xffffffffu, M, o));
      if (lane == 0) sm.Mt[task] = M;
      const double2 z = valid ? a.z[k] : make_double2(0, 1);
      const double2 wr = (valid && a.has_rho) ? a.w_rho[k] : make_double2(0, 0);
      const double2 we = (valid && a.has_edm) ? a.w_edm[k] : make_double2(0, 0);
      double2 Q = make_double2(0, 0);
      double lacc = 0.0;
      for (int g = (M - 1) / CK; M > 0 && g >= 0; --g) {
        const int m0 = g * CK, mend = min(m0 + CK, M);
        const int lim = min(mend, nkk);
        if (valid && m0 < nkk) {
          const size_t ce = ((size_t)g * RK + e) * 2;
          double2 cur = ck[ce], prev = ck[ce + 1];
          buf[e] = cur;
          for (int mm = m0; mm < lim; ++mm) {
            const double* h = hc + ((size_t)mm * R + cc) * 3;
            const double2 nxt = real_step(cur, prev, h[0], h[1], h[2], z);
            prev = cur;
            cur = nxt;
            buf[(size_t)(mm + 1 - m0) * RK + e] = nxt;
          }
        }
        for (int mm = mend - 1; mm >= m0; --mm) {
          double2 cm = make_double2(0, 0);
          if (valid && mm < nkk) {
            const double c1 = hc[((size_t)mm * R + cc) * 3];
            const double2 pm = buf[(size_t)(mm - m0) * RK + e], pn = buf[(size_t)(mm + 1 - m0) * RK + e];
            const double2 d = cmul(pm, pn);
            const double f = 1.0 / (c1 * cabs2(d));
            if (f > 0.0) {  // a product beyond the FP64 range adds nothing
              Q.x = fma(d.x, f, Q.x);
              Q.y = fma(-d.y, f, Q.y);
            }
            cm = cscale(cmul(pm, Q), c1 * c1);
          }
          lacc = fma(cm.y, ht[(size_t)mm * R + cc], lacc);
          if (cgs && valid) cgs[((size_t)mm * R + cc) * K + k] = cm;
          // v is real: only Im(w y) reaches rho and P^E
          double vr = fma(wr.x, cm.y, wr.y * cm.x), ve = fma(we.x, cm.y, we.y * cm.x);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            vr += __shfl_xor_sync(0xffffffffu, vr, o);
            ve += __shfl_xor_sync(0xffffffffu, ve, o);
          }
          if (lane == 0) {
            const size_t pe = (((size_t)mm * R + cc) * KG + kg) * 2;
            cp[pe] = vr;
            cp[pe + 1] = ve;
          }
        }
      }
      if (valid) {
        const long long col = (long long)sm.panel * a.C + cc;
        const long long o = (long long)k * a.nrhs + col;
        if (a.ldos) a.ldos[o] = -lacc / 3.141592653589793238462643383279502884;
        if (a.resid) a.resid[o] = resk[e];
        if (a.conv) a.conv[o] = resk[e] <= a.tol ? 1 : 0;
      }
    }
    __syncthreads();
    if (tid < R) {
      int mc = 0;
      for (int g = 0; g < KG; ++g) mc = max(mc, sm.Mt[tid * KG + g]);
      sm.Mc[tid] = mc;
    }
    __syncthreads();
  }
  // F2: C_m = sum over shift groups
  if (a.has_rho || a.has_edm) {
    int mmax = 0;
    for (int i = 0; i < R; ++i) mmax = max(mmax, sm.Mc[i]);
    for (int e = tid; e < mmax * R; e += tpb()) {
      const int m = e / R, cc = e - m * R;
      if (m >= sm.Mc[cc]) continue;
      double sr = 0.0, se = 0.0;
      for (int g = 0; g < KG; ++g) {
        if (m >= sm.Mt[cc * KG + g]) continue;
        const size_t pe = (((size_t)m * R + cc) * KG + g) * 2;
        sr += cp[pe];
        se += cp[pe + 1];
      }
      cf[((size_t)m * R + cc) * 2] = sr;
      cf[((size_t)m * R + cc) * 2 + 1] = se;
    }
    __syncthreads();
    // F3: rho_ij = sum_m C^rho_m v_m[i], edm_ij likewise
    const int Mt_ = sm.off[R];
    for (int e = tid; e < Mt_; e += tpb()) {
      int cc = 0;
      while (sm.off[cc + 1] <= e) ++cc;
      const int t = e - sm.off[cc];
      double xr = 0.0, xe = 0.0;
      for (int m = 0; m < sm.Mc[cc]; ++m) {
        const double rv = hr[(size_t)m * a.Mcap + e];
        xr = fma(cf[((size_t)m * R + cc) * 2], rv, xr);
        xe = fma(cf[((size_t)m * R + cc) * 2 + 1], rv, xe);
      }
      const long long o = a.out_off[(long long)sm.panel * a.C + cc] + t;
      if (a.rho && a.has_rho) a.rho[o] = xr;
      if (a.edm && a.has_edm) a.edm[o] = xe;
    }
    __syncthreads();
  }
  // F4: per-column outputs
  if (tid < R && sm.mc[tid] > 0) {
    const long long col = (long long)sm.panel * a.C + tid;
    const int base = a.m.row_ptr[sm.j[tid]];
    if (a.has_rho && a.rho && (a.q || a.e_loc)) {
      double qs = 0.0, es = 0.0;
      for (int t = 0; t < sm.mc[tid]; ++t) {
        const double rv = a.rho[a.out_off[col] + t];
        qs = fma(rv, a.m.s_val[base + t], qs);
        es = fma(rv, a.m.h_val[base + t], es);
      }
      if (a.q) a.q[col] = qs;
      if (a.e_loc) a.e_loc[col] = es;
    }
    if (a.iters) a.iters[col] = sm.nc[tid];
    if (a.inner_iters) a.inner_iters[col] = sm.inner_count;
    int st = sm.cst[tid] | sm.st[tid >> 1] | (sm.bc_fail ? kStTimeout : 0);
    for (int k = 0; k < K; ++k)
      if (!(resk[tid * K + k] <= a.tol)) st |= kStNoConv;
    a.status[col] = st;
    if (a.col_status) a.col_status[col] = st;
  }
  if (cgs && a.g_proj) {
    __syncthreads();
    const int Mt_ = sm.off[R];
    for (int e = tid; e < Mt_ * K; e += tpb()) {
      const int k = e / Mt_, f = e - k * Mt_;
      int cc = 0;
      while (sm.off[cc + 1] <= f) ++cc;
      const int nkk = nk[cc * K + k];
      double2 g = make_double2(0, 0);
      for (int m = 0; m < nkk; ++m) {
        const double2 y = cgs[((size_t)m * R + cc) * K + k];
        const double rv = hr[(size_t)m * a.Mcap + f];
        g.x = fma(y.x, rv, g.x);
        g.y = fma(y.y, rv, g.y);
      }
      a.g_proj[(long long)k * a.P + a.out_off[(long long)sm.panel * a.C + cc] + f - sm.off[cc]] = g;
    }
  }
  __syncthreads();
}

}  // namespace gbk
