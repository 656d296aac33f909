// Direct Runge-Kutta stage for FP64, for WENO5, and for FP32 UW3 grids without the packed layout (a
// ragged n_phi, or too small for a staged box).  Same stage as stage_kernel (vlb_stage.cu); the populations
// are read straight from global memory through L1 instead of being staged, so a tile can be small.
//
// FP64 is bound by the FP64 units (1.25 TFLOP/s nominal, pipe 99% active on the busiest SM): what counts is
// the number of FP64 operations (780 a node and stage in the staged kernel, 500-550 here: parity basis
// and row table of vlb_node.cuh, folded centre taps) and their spread over all SMs (16 x 32 tiles left 56 of 152
// SMs idle on 128 x 384, and 148 on 32 x 64).  Per step: 32 x 64 304 -> 35 us, 128 x 384 305 -> 175 us.  FP64 CTAs
// of one thread per node do not trigger the next stage early: its CTAs would fill the free slots of
// lightly loaded SMs and unbalance it (85 us a stage against 66 on 128 x 384).
// FP32 grids off the packed layout are bound by latency (one wave); no staging with a modulo and a
// 4-byte copy per element: 250 x 501 diffusive 57.6 -> 39 us per step.
// WENO5 is bound by issue (about 50 instructions a face): a face is evaluated once for both its nodes instead
// of once for each, with one approximate reciprocal instead of four divisions.  FP32, 256 x 512: 132 -> 72 us
// per step (83 with the range check as a branch in every face); FP64, 128 x 256: 2399 -> 513 us.  At most 102
// registers (five CTAs per SM): with seven and spills 75 us at 256 x 512, 517 against 537 us at 1024 x 1024.
#include "vlb_node.cuh"

namespace vlb {

namespace {

__device__ const RowRules<float> g_rules32 = make_row_rules<float>();
__device__ const RowRules<double> g_rules64 = make_row_rules<double>();
template <typename T>
__device__ __forceinline__ const RowRule<T>& row_rules(int e) {
  if constexpr (sizeof(T) == 8)
    return g_rules64.e[e];
  else
    return g_rules32.e[e];
}

template <typename T>
struct DirectConst {
  NodeConst<T> nc;
  T v[4], K[4][4], ww[4][4];
};

// Element at byte offset `off` of an array whose base is uniform over the CTA.
template <typename T, typename Off>
__device__ __forceinline__ T at(const T* base, Off off) {
  return *reinterpret_cast<const T*>(reinterpret_cast<const char*>(base) + off);
}
template <typename T, typename Off>
__device__ __forceinline__ void put(T* base, Off off, T v) {
  *reinterpret_cast<T*>(reinterpret_cast<char*>(base) + off) = v;
}

__device__ __forceinline__ int wrap_near(int x, int n) {  // -n <= x
  if (x < 0) return x + n;
  while (x >= n) x -= n;
  return x;
}

// Moment-box slots of a TQ x TSW tile: the tile's nodes, then one halo row on each side, then one halo
// column on each side (no corners).
template <int TQ, int TSW>
__device__ __forceinline__ void slot_node(int it, int& mr, int& mc) {
  if (it < TQ * TSW) {
    mr = 1 + it / TSW;
    mc = 1 + it % TSW;
  } else if (it < TQ * TSW + 2 * TSW) {
    const int j = it - TQ * TSW;
    mr = j < TSW ? 0 : TQ + 1;
    mc = 1 + j % TSW;
  } else {
    const int j = it - TQ * TSW - 2 * TSW;
    mr = 1 + j % TQ;
    mc = j < TQ ? 0 : TSW + 1;
  }
}

// One CTA per TQ x TSW tile.  Step 1 puts the moments and mu of the tile and a halo of 1 into shared memory
// (dn, 1/n, u^theta, u^phi, mu); step 2 evaluates the right-hand side and the update.  Off: the type of a byte offset
// within one array.
template <typename T, int ADV, int CH, bool F0, int TQ, int TSW, bool SPLIT, typename Off>
__global__ void __launch_bounds__(TQ* TSW*(SPLIT ? 4 : 1), ADV == VLB_WENO5 && sizeof(T) == 4 ? 5 : 0)
    direct_kernel(StageArgs<T> a, const __grid_constant__ DirectConst<T> dc) {
  constexpr bool DF = sizeof(T) == 4;
  constexpr int MS = TSW + 2, MN = (TQ + 2) * MS, NTH = TQ * TSW * (SPLIT ? 4 : 1);
  constexpr int ITEMS = TQ * TSW + 2 * TSW + 2 * TQ;
  constexpr bool HOLD = sizeof(T) == 8 && ADV == VLB_UW3;  // hold U^n in registers over step 1
  constexpr bool TAB = !SPLIT && sizeof(T) == 8;  // row table in shared memory (FP64-bound), else per thread
  constexpr int NE = row_entries<T>(), RP = NE | 1;  // odd row pitch: two rows of a warp on different banks
  __shared__ T s_dn[MN], s_in[MN], s_ut[MN], s_up[MN], s_mu[MN], s_rt[TAB ? TQ * RP : 1];
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  const int nt = a.nt, ns = a.ns, tid = threadIdx.x;
  const int tiles_s = (ns + TSW - 1) / TSW;  // 1-D grid: a column grid has more tile rows than gridDim.y may hold
  const int q0 = (int)(blockIdx.x / tiles_s) * TQ, s0 = (int)(blockIdx.x % tiles_s) * TSW;
  const int64_t st = a.stride;
  constexpr Off B = sizeof(T);
  const NodeConst<T>& nc = dc.nc;
  const T* phi = a.fin + NPOP * st;
  constexpr bool KEEP = !SPLIT && ADV == VLB_UW3;  // the parity combinations stay in registers for step 2
  T P[SPLIT ? 1 : 16], U0[SPLIT ? 4 : 16];
  if (F0) {  // U^n of this thread's populations, in flight over step 1
    const int node = SPLIT ? tid >> 2 : tid, q = q0 + node / TSW, s = s0 + node % TSW;
    if (HOLD && q < nt && s < ns)
#pragma unroll
      for (int k = 0; k < (SPLIT ? 4 : 16); ++k)
        U0[k] = SPLIT ? a.f0[(k + 4 * (tid & 3)) * st + (int64_t)q * ns + s]
                      : at(a.f0 + k * st, B * (uint32_t)(q * ns + s));
  }
  if constexpr (TAB) {
    for (int e = tid; e < TQ * NE; e += NTH)
      if (q0 + e / NE < nt) s_rt[(e / NE) * RP + e % NE] = row_entry(row_rules<T>(e % NE), a, q0 + e / NE, e % NE >= E_CC);
  }

  auto moments = [&](int it, bool keep) {
    int mr, mc;
    slot_node<TQ, TSW>(it, mr, mc);
    if (q0 + mr - 1 > nt || s0 + mc - 1 > ns) return;  // beyond the halo of the last node
    const int q = wrap_near(q0 + mr - 1, nt), s = wrap_near(s0 + mc - 1, ns);
    const Off id = B * (uint32_t)(q * ns + s);
    T g[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) g[k] = at(a.fin + k * st, id);
    const Off in_ = B * (uint32_t)((q + 1 < nt ? q + 1 : 0) * ns + s);
    const Off is = B * (uint32_t)((q > 0 ? q - 1 : nt - 1) * ns + s);
    const Off ie = B * (uint32_t)(q * ns + (s + 1 < ns ? s + 1 : 0));
    const uint32_t iw = B * (uint32_t)(q * ns + (s > 0 ? s - 1 : ns - 1));
    const T ph = at(phi, id);
    T dN = vsub(at(phi, in_), ph), dS = vsub(ph, at(phi, is)), lo = T(0);
    T dE = vsub(at(phi, ie), ph), dW = vsub(ph, at(phi, iw));
    if constexpr (DF) {
      const T* pl = phi + st;
      lo = at(pl, id);
      dN = vadd(dN, vsub(at(pl, in_), lo));
      dS = vadd(dS, vsub(lo, at(pl, is)));
      dE = vadd(dE, vsub(at(pl, ie), lo));
      dW = vadd(dW, vsub(lo, at(pl, iw)));
    }
    const T lt = a.coef[C_LT * nt + q], lp = a.coef[C_LP * nt + q];
    const T jp = a.coef[C_JP * nt + q], jm = a.coef[C_JM * nt + q];
    to_parity16(g);
    T dn, mt, mp;
    parity_moments(g, nc, dn, mt, mp);
    const T inv_n = node_recip(vadd(a.n0, dn));
    const int mi = mr * MS + mc;
    s_dn[mi] = dn;
    s_in[mi] = inv_n;
    s_ut[mi] = node_velocity(mt, inv_n, nc.fix);
    s_up[mi] = node_velocity(mp, inv_n, nc.fix);
    const T lap = vfma(lp, vsub(dE, dW), vmul(lt, vsub(vmul(jp, dN), vmul(jm, dS))));
    const T ph2 = vmul(ph, ph);
    T cubic = vmul(ph, vsub(T(1), ph2));
    if constexpr (DF) cubic = vfma(vsub(T(1), vmul(T(3), ph2)), lo, cubic);  // at hi + lo, to first order in lo
    s_mu[mi] = vsub(vmul(-a.A, cubic), vmul(a.kappa, lap));
    if constexpr (KEEP) {
      if (keep)
#pragma unroll
        for (int k = 0; k < 16; ++k) P[k] = g[k];
    }
  };
  if constexpr (!SPLIT) {
    moments(tid, true);
    for (int it = NTH + tid; it < ITEMS; it += NTH) moments(it, false);
  } else {
    for (int it = tid; it < ITEMS; it += NTH) moments(it, false);
  }
  __syncthreads();
  if (SPLIT || sizeof(T) == 4) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");

  constexpr bool WENO = ADV == VLB_WENO5;
  __shared__ T s_adv[WENO ? 16 * TQ * TSW : 1], s_edge[WENO ? 16 * TQ : 1];
  if constexpr (WENO) {
    // Advection: -dt v (face difference) along both directions.  Warp i takes the four populations of theta
    // velocity v_i, a lane a column.  Everything is seen from the upwind side (up = -1 for v > 0, +1 for
    // v < 0), so that one face formula serves both signs.  Along theta a lane marches over the tile's rows,
    // so a face is evaluated once for its two nodes (TQ + 1 faces for TQ nodes); along varphi a lane
    // evaluates its downwind face and takes the upwind one from its neighbour, the tile's first lane from
    // a face formed beforehand.
    static_assert(!SPLIT && TSW == 32 && NTH == 4 * 32 && 16 * TQ <= NTH, "a warp per theta velocity");
    const int i = tid >> 5, lane = tid & 31;
    auto near = [](int x, int n) {
      while (x < 0) x += n;
      while (x >= n) x -= n;
      return x;
    };
    auto col = [&](int c) { return B * (uint32_t)near(s0 + c, ns); };
    bool bad = false;
    if (tid < 16 * TQ) {  // the tile's first upwind face: at s0 - 1/2 (v > 0) or s0 + TSW - 1/2
      const int k = tid / TQ, dn = (k & 3) >= 2 ? 1 : -1, first = dn > 0 ? -1 : TSW;
      const Off row = B * (uint32_t)(wrap_near(q0 + tid % TQ, nt) * ns);
      T x[5];
#pragma unroll
      for (int d = 0; d < 5; ++d) x[d] = at(a.fin + k * st, row + col(first + dn * (d - 2)));
      s_edge[tid] = weno5_face(x[0], x[1], x[2], x[3], x[4], bad);
    }
    __syncthreads();
    const int dt_ = i >= 2 ? 1 : -1, top = i >= 2 ? 0 : TQ - 1;  // downwind step along theta; the first row of the march
    Off ro[TQ + 5], cs[5];  // rows of the march, columns lane - 2 .. lane + 2 (byte offsets)
    T J[TQ + 5];
#pragma unroll
    for (int d = 0; d < TQ + 5; ++d) {
      const int row = near(q0 + top + dt_ * (d - 3), nt);
      ro[d] = B * (uint32_t)(row * ns);
      J[d] = a.coef[(int64_t)C_J * nt + row];
    }
#pragma unroll
    for (int d = 0; d < 5; ++d) cs[d] = col(lane + d - 2);
    T vct[TQ], ccp[TQ];
#pragma unroll
    for (int r = 0; r < TQ; ++r) {
      const int row = near(q0 + top + dt_ * r, nt);
      vct[r] = -(dt_ > 0 ? dc.v[i] : -dc.v[i]) * (a.coef[(int64_t)C_CT * nt + row] * a.dt);
      ccp[r] = a.coef[(int64_t)C_CP * nt + row] * a.dt;
    }
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
      const int k = 4 * i + j;
      const T* f = a.fin + k * st;
      const T fref = a.n0 * dc.ww[i][j];  // theta reconstructs the full J f
      const int dp = j >= 2 ? 1 : -1;     // downwind step along varphi
      const T vj = dp > 0 ? dc.v[j] : -dc.v[j];
      const Off c0 = dp > 0 ? cs[0] : cs[4], c1 = dp > 0 ? cs[1] : cs[3], c3 = dp > 0 ? cs[3] : cs[1];
      const Off c4 = dp > 0 ? cs[4] : cs[0];
      T G[TQ + 5], x[TQ];
#pragma unroll
      for (int d = 0; d < TQ + 5; ++d) {
        const T g = at(f, ro[d] + cs[2]);
        if (d >= 3 && d < TQ + 3) x[d - 3] = g;
        G[d] = J[d] * (g + fref);
      }
      T last = weno5_face(G[0], G[1], G[2], G[3], G[4], bad);
#pragma unroll
      for (int r = 0; r < TQ; ++r) {
        const int lrow = top + dt_ * r;
        const T F = weno5_face(G[r + 1], G[r + 2], G[r + 3], G[r + 4], G[r + 5], bad);
        T adv = vct[r] * (F - last);  // -|v| (downwind - upwind face) in both directions
        last = F;
        const Off o = ro[r + 3];
        const T Fd = weno5_face(at(f, o + c0), at(f, o + c1), x[r], at(f, o + c3), at(f, o + c4), bad);
        T Fu = __shfl_sync(0xffffffffu, Fd, (lane - dp) & 31);
        if (lane == (dp > 0 ? 0 : 31)) Fu = s_edge[k * TQ + lrow];
        adv -= vj * ccp[r] * (Fd - Fu);
        s_adv[(k * TQ + lrow) * TSW + lane] = adv;
      }
    }
    if (__syncthreads_or(bad)) {  // rare: the whole tile again with the plain face formula
#pragma unroll 1
      for (int x = lane; x < 4 * TQ * TSW; x += 32) {
        const int j = x / (TQ * TSW), lrow = x / TSW % TQ, k = 4 * i + j, row = near(q0 + lrow, nt);
        const T* f = a.fin + k * st;
        T xt[7], xp[7];
#pragma unroll
        for (int d = 0; d < 7; ++d) {
          const int rd = near(q0 + lrow + d - 3, nt);
          xt[d] = a.coef[(int64_t)C_J * nt + rd] * (at(f, B * (uint32_t)(rd * ns) + cs[2]) + a.n0 * dc.ww[i][j]);
          xp[d] = at(f, B * (uint32_t)(row * ns) + col(lane + d - 3));
        }
        const T Dt = i >= 2 ? weno_diff<T, true>(xt) : weno_diff<T, false>(xt);
        const T Dp = j >= 2 ? weno_diff<T, true>(xp) : weno_diff<T, false>(xp);
        s_adv[(k * TQ + lrow) * TSW + lane] = -(dc.v[i] * (a.coef[(int64_t)C_CT * nt + row] * a.dt)) * Dt -
                                              (dc.v[j] * (a.coef[(int64_t)C_CP * nt + row] * a.dt)) * Dp;
      }
      __syncthreads();
    }
  }

  const int node = SPLIT ? tid >> 2 : tid;
  const int lr = node / TSW, lc = node % TSW;
  const int q = q0 + lr, s = s0 + lc;
  if (q >= nt || s >= ns) return;
  const int mi = (lr + 1) * MS + lc + 1;
  T rl[TAB ? 1 : NE];
  if constexpr (!TAB) row_all<T>(rl, a, q);
  const T* rt = TAB ? s_rt + lr * RP : rl;
  const Off id = B * (uint32_t)(q * ns + s);  // byte offsets within one array (launch_direct checks the range)
  const int qn = q + 1 < nt ? q + 1 : 0, qs = q > 0 ? q - 1 : nt - 1;
  const int qnn = wrap_near(q + 2, nt), qss = wrap_near(q - 2, nt);
  const int se = s + 1 < ns ? s + 1 : 0, sw = s > 0 ? s - 1 : ns - 1;
  const int see = wrap_near(s + 2, ns), sww = s >= 2 ? s - 2 : (s - 2 + 2 * ns) % ns;
  const T dt = a.dt, itau = a.inv_tau * dt;
  const T dn = s_dn[mi], ut = s_ut[mi], up = s_up[mi], ph = at(phi, id);
  const T mu_c = s_mu[mi], mu_n = s_mu[mi + MS], mu_s = s_mu[mi - MS], mu_e = s_mu[mi + 1], mu_w = s_mu[mi - 1];
  T Ft = T(0), Fp = T(0);  // times dt
  if (CH == VLB_HYDRO) {   // n F = -phi grad mu (Eq. pbin), central differences
    const T pn = vmul(ph, s_in[mi]);
    Ft = vmul(vmul(pn, vsub(mu_s, mu_n)), a.gt * dt);
    Fp = vmul(vmul(pn, vsub(mu_w, mu_e)), rt[E_GP]);
  }
  const Off on = B * (uint32_t)(qn * ns + s), os = B * (uint32_t)(qs * ns + s);
  const Off onn = B * (uint32_t)(qnn * ns + s), oss = B * (uint32_t)(qss * ns + s);
  const Off oe = B * (uint32_t)(q * ns + se), ow = B * (uint32_t)(q * ns + sw);
  const Off oee = B * (uint32_t)(q * ns + see), oww = B * (uint32_t)(q * ns + sww);
  const int i_split = SPLIT ? tid & 3 : 0;
  if (!SPLIT || i_split == 0) {
    // Cahn-Hilliard: M Delta mu - div(u phi) (Eq. CH), flux form with mean face values, times dt
    T L = vmul(rt[E_LP], vadd(vsub(mu_e, mu_c), vsub(mu_w, mu_c)));
    L = vfma(rt[E_LT], vfma(rt[E_JP], vsub(mu_n, mu_c), vmul(rt[E_JM], vsub(mu_s, mu_c))), L);
    if (CH == VLB_HYDRO) {
      L = vfma(-rt[E_XN], vmul(s_ut[mi + MS], at(phi, on)), L);
      L = vfma(rt[E_XS], vmul(s_ut[mi - MS], at(phi, os)), L);
      L = vfma(-rt[E_YP], vsub(vmul(s_up[mi + 1], at(phi, oe)), vmul(s_up[mi - 1], at(phi, ow))), L);
    }
    if (a.dphi) {
      put(a.dphi, id, L);  // the stabilised Cahn-Hilliard solve forms phi
    } else {
      const T lo = DF ? at(phi + st, id) : T(0);
      T base = ph, base_lo = lo, inc = L;
      if (F0) {
        base = at(a.f0 + NPOP * st, id);
        base_lo = DF ? at(a.f0 + (NPOP + 1) * st, id) : T(0);
        inc = vmul(a.b, vadd(vadd(vsub(ph, base), vsub(lo, base_lo)), L));
      }
      if constexpr (DF) {  // (hi, lo) <- (base, base_lo) + inc, an error-free sum, renormalised
        const T s1 = vadd(base, inc), bb = vsub(s1, base);
        const T lo2 = vadd(base_lo, vadd(vsub(base, vsub(s1, bb)), vsub(inc, bb)));
        const T hi = vadd(s1, lo2);
        put(a.fout + NPOP * st, id, hi);
        put(a.fout + (NPOP + 1) * st, id, vsub(lo2, vsub(hi, s1)));
      } else {
        put(a.fout + NPOP * st, id, vadd(base, inc));
      }
    }
  }

  // population k: acc (dt times the other terms) -> stored update.  UW3 seen from the upwind side has the
  // weights 1, -6, 3, 2 on the far, near, centre and downwind nodes (tf .. td: theta, on J g; pv: varphi).
  // FP64 folds the three centre taps into one coefficient, whose rounding is far below the scheme's.
  // FP32 keeps the varphi difference on whole-number weights, which cancel on a uniform field, and takes the theta
  // taps on differences to the node, with their sum as the coefficient tm: they nearly cancel, so the products
  // stay small (tau = 0.1, 401 x 63: 1.05e-7 -> 0.96e-7; 250 x 501, 8 steps: 314 -> 308 us).
  auto update = [&](int k, T acc, T g0, T tf, T tn, T tm, T td, Off rf, Off rn, Off rd, int y, T cc,
                    Off cf, Off cn, Off cd) {
    const T* f = a.fin + k * st;
    const T g = at(f, id), pv = rt[E_TH + 8 * y + TAP_PV];
    if (F0 && !HOLD) g0 = at(a.f0 + k * st, id);
    if (F0) acc = vadd(acc, vsub(g, g0));
    if constexpr (!WENO) {
      if constexpr (DF) {
        acc = vfma(tf, vsub(at(f, rf), g), acc);
        acc = vfma(tn, vsub(at(f, rn), g), acc);
        acc = vfma(td, vsub(at(f, rd), g), acc);
      } else {
        acc = vfma(tf, at(f, rf), acc);
        acc = vfma(tn, at(f, rn), acc);
        acc = vfma(td, at(f, rd), acc);
      }
    }
    if constexpr (WENO) {
      acc = vadd(acc, s_adv[(k * TQ + lr) * TSW + lc]);
      acc = vfma(-itau, g, acc);
    } else if constexpr (DF) {
      acc = vfma(tm, g, acc);
      const T D = vfma(T(2), at(f, cd), vfma(T(3), g, vfma(T(-6), at(f, cn), at(f, cf))));
      acc = vfma(-pv, D, acc);
      acc = vfma(-itau, g, acc);
    } else {
      acc = vfma(-pv, at(f, cf), acc);
      acc = vfma(rt[E_PV6 + y], at(f, cn), acc);
      acc = vfma(rt[E_PV2 + y], at(f, cd), acc);
      acc = vfma(cc, g, acc);
    }
    put(a.fout + k * st, id, F0 ? vfma(a.b, acc, g0) : vadd(acc, g));
  };

  if constexpr (!SPLIT) {
    T R[16];
    if constexpr (!KEEP) {
#pragma unroll
      for (int k = 0; k < 16; ++k) P[k] = at(a.fin + k * st, id);
      to_parity16(P);
    }
    velocity_space(P, R, nc, rt, Ft, Fp, itau, a.n0, dn, ut, up);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int x = (i == 0 || i == 3) ? 0 : 1;
      const T* t = rt + E_TH + 8 * x;
      const T tf = t[i >= 2 ? TAP_FARP : TAP_FARN], tn = t[i >= 2 ? TAP_NEARP : TAP_NEARN];
      T tm = t[TAP_MID];
      if constexpr (DF) {  // the sum of the four taps, v_i (E + Gamma)
        const T gv = x == 0 ? rt[E_GBB] * (T(1) / nc.v[0]) : rt[E_GAA] * (T(1) / nc.v[1]);
        tm = vadd(vfma(i >= 2 ? nc.v[x] : -nc.v[x], rt[E_EM], rt[E_NEB + x]), i >= 2 ? gv : -gv);
      }
      const T td = t[i >= 2 ? TAP_DOWNP : TAP_DOWNN];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int y = (j == 0 || j == 3) ? 0 : 1;
        update(4 * i + j, R[4 * i + j], U0[4 * i + j], tf, tn, tm, td, i >= 2 ? oss : onn, i >= 2 ? os : on,
               i >= 2 ? on : os, y, DF ? T(0) : rt[E_CC + 2 * x + y], j >= 2 ? oww : oee, j >= 2 ? ow : oe,
               j >= 2 ? oe : ow);
      }
    }
  } else {
    // four threads per node, thread i the populations of theta velocity v_i
    const int i = i_split, x = (i == 0 || i == 3) ? 0 : 1;
    const bool pos = i >= 2;
    const T vi = dc.v[i], Ki[4] = {dc.K[i][0], dc.K[i][1], dc.K[i][2], dc.K[i][3]};
    T dvt[4], h[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) dvt[j] = vmul(Ki[0], at(a.fin + j * st, id));
#pragma unroll
    for (int m = 1; m < 4; ++m)
#pragma unroll
      for (int j = 0; j < 4; ++j) dvt[j] = vfma(Ki[m], at(a.fin + (4 * m + j) * st, id), dvt[j]);
    // Gamma v_i v_m from the row's products of magnitudes
    T gb = x == 0 ? rt[E_GBB] : rt[E_GBA], ga = x == 0 ? rt[E_GBA] : rt[E_GAA];
    gb = pos ? gb : -gb;
    ga = pos ? ga : -ga;
    h[0] = vmul(vsub(gb, Fp), at(a.fin + (4 * i) * st, id));
    h[1] = vmul(vsub(ga, Fp), at(a.fin + (4 * i + 1) * st, id));
    h[2] = vmul(vsub(-ga, Fp), at(a.fin + (4 * i + 2) * st, id));
    h[3] = vmul(vsub(-gb, Fp), at(a.fin + (4 * i + 3) * st, id));
    const T cyb = vsub(rt[E_GBB], Ft), cya = vsub(rt[E_GAA], Ft);
    const T hu = vmul(T(-0.5), vfma(ut, ut, vmul(up, up))), c0 = vadd(T(1), hu);
    const T dntau = vmul(dn, itau), ntau = vfma(itau, a.n0, dntau), ai = vmul(vi, ut);
    // n0 v_i (E(sign v_i) + F^theta): the odd part changes sign with v_i, the even part does not
    const T ci = vadd(dntau, vmul(a.n0, vadd(x == 0 ? rt[E_NEB] : rt[E_NEA], vmul(vi, vadd(rt[E_EM], Ft))))), pF = vmul(a.n0, Fp);
    const T vc = vmul(pos ? vi : -vi, vmul(a.coef[(int64_t)C_CT * nt + q], dt * T(1.0 / 6.0)));
    const T* J = a.coef + (int64_t)C_J * nt;
    const T tf = -vmul(vc, J[pos ? qss : qnn]), tn = vmul(T(6) * vc, J[pos ? qs : qn]);
    const T td = vmul(T(-2) * vc, J[pos ? qn : qs]), tm = vmul(T(-3) * vc, J[q]);
    const T ccx = vsub(tm, itau);
    const Off rf = pos ? oss : onn, rn = pos ? os : on, rd = pos ? on : os;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int y = (j == 0 || j == 3) ? 0 : 1;
      T acc = vmul(dc.K[j][0], h[0]);
#pragma unroll
      for (int m = 1; m < 4; ++m) acc = vfma(dc.K[j][m], h[m], acc);
      acc = vfma(y == 0 ? cyb : cya, dvt[j], acc);
      const T xi = vfma(dc.v[j], up, ai);
      const T pm1 = vfma(xi, vfma(xi, vfma(xi, T(1.0 / 6.0), T(0.5)), c0), hu);
      acc = vfma(dc.ww[i][j], vfma(ntau, pm1, vfma(dc.v[j], pF, ci)), acc);
      update(4 * i + j, acc, U0[j], tf, tn, tm, td, rf, rn, rd, y, DF ? T(0) : vfma(T(-3), rt[E_TH + 8 * y + TAP_PV], ccx),
             j >= 2 ? oww : oee, j >= 2 ? ow : oe, j >= 2 ? oe : ow);
    }
  }
}

template <typename T>
DirectConst<T> make_direct_const() {
  const VelocityConsts d = velocity_consts();
  DirectConst<T> c;
  c.nc = make_node_const<T>();
  for (int i = 0; i < 4; ++i) {
    c.v[i] = (T)d.v[i];
    for (int m = 0; m < 4; ++m) {
      c.K[i][m] = (T)d.K[i][m];
      c.ww[i][m] = (T)(d.w[i] * d.w[m]);
    }
  }
  return c;
}

template <typename T, int ADV, int CH, bool F0, int TQ, int TSW, bool SPLIT, typename Off = uint32_t>
cudaError_t launch_direct_t(const StageArgs<T>& a, cudaStream_t st) {
  static const DirectConst<T> dc = make_direct_const<T>();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((a.ns + TSW - 1) / TSW) * (unsigned)((a.nt + TQ - 1) / TQ));
  cfg.blockDim = dim3(TQ * TSW * (SPLIT ? 4 : 1));
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, direct_kernel<T, ADV, CH, F0, TQ, TSW, SPLIT, Off>, a, dc);
}

// FP32: 4 x 32 tiles, one thread per node (8 x 32 tiles with 64 registers: 316 us against 304-320 on eight
// steps of 250 x 501, within the spread).  FP64: 8 x 16 tiles, one thread per node, four warps a CTA: an SM
// retires one FP64 warp instruction in 19 cycles, but a lone warp only one in 64 (measured), so four
// warps saturate it and below about 32 nodes per SM the time is one warp's chain; there four
// threads share a node (2 x 8 nodes a CTA).  Per step, one / four threads a node: 32 x 64 72 / 34 us, 64 x 128
// 72 / 93 us, 128 x 384 175 / 330 us.
constexpr int64_t kSplitNodes = 32 * 152;
// Byte offsets within one array are 32 bits up to 2^32 bytes.  An FP32 array cannot be larger (its grid would need
// 360 GB: 352 bytes a node with the staging area); FP64 grids of 2^29 nodes and more take 64-bit offsets (544 bytes a
// node: 272 GiB, which the device holds up to about 547 million nodes).
constexpr uint64_t kWideNodes = (uint64_t)1 << 29;

template <typename T, int ADV, int CH, bool F0>
cudaError_t launch_direct_v(const StageArgs<T>& a, cudaStream_t st) {
  if constexpr (sizeof(T) == 8) {
    if ((uint64_t)a.nt * a.ns >= kWideNodes || (a.route & VLB_TEST_WIDE_OFFSETS))
      return launch_direct_t<T, ADV, CH, F0, ADV == VLB_WENO5 ? 4 : 8, ADV == VLB_WENO5 ? 32 : 16, false, uint64_t>(a, st);
  }
  if constexpr (ADV == VLB_WENO5 || sizeof(T) == 4) {
    return launch_direct_t<T, ADV, CH, F0, 4, 32, false>(a, st);
  } else {
    if ((int64_t)a.nt * a.ns <= kSplitNodes) return launch_direct_t<T, ADV, CH, F0, 2, 8, true>(a, st);
    return launch_direct_t<T, ADV, CH, F0, 8, 16, false>(a, st);
  }
}

template <typename T, int ADV>
cudaError_t launch_direct_a(const StageArgs<T>& a, int ch_mode, cudaStream_t st) {
  if (ch_mode == VLB_HYDRO)
    return a.f0 ? launch_direct_v<T, ADV, VLB_HYDRO, true>(a, st) : launch_direct_v<T, ADV, VLB_HYDRO, false>(a, st);
  return a.f0 ? launch_direct_v<T, ADV, VLB_DIFFUSIVE, true>(a, st)
              : launch_direct_v<T, ADV, VLB_DIFFUSIVE, false>(a, st);
}

}  // namespace

template <typename T>
cudaError_t launch_direct(const StageArgs<T>& a, int advection, int ch_mode, cudaStream_t st) {
  return advection == VLB_UW3 ? launch_direct_a<T, VLB_UW3>(a, ch_mode, st) : launch_direct_a<T, VLB_WENO5>(a, ch_mode, st);
}

template cudaError_t launch_direct<float>(const StageArgs<float>&, int, int, cudaStream_t);
template cudaError_t launch_direct<double>(const StageArgs<double>&, int, int, cudaStream_t);

}  // namespace vlb
