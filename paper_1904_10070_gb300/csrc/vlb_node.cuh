// Per-node arithmetic shared by the step kernels: the velocity-space part of the right-hand side
// (force, inertial and BGK terms of Eq. boltz_tor) in the parity basis of the velocity set.
//
// The Q = 4 velocities come in pairs +-b, +-a (b = v_4, a = v_3), so each velocity direction splits
// into even and odd combinations c = 0..3: E_b = g_+b + g_-b, E_a, O_b = g_+b - g_-b, O_a.  The
// derivative kernel K^H changes the sign of the velocity under reflection, so it maps even to odd and
// odd to even: 8 multiplications instead of 16 per vector.  The Hermite equilibrium splits likewise
// into even-even, odd-even, even-odd and odd-odd parts of a few operations each.  One node costs 32 (to the
// basis) + 32 (back) additions and about 180 multiply-adds, against about 330 on the populations
// themselves; the step kernels are bound by the floating-point units, so this is their main saving.
// Moments are sums of the same combinations.
//
// V is the lane type: double, float, or float2 (two nodes in packed FP32x2 arithmetic).  The
// operations of the UW3 step are explicitly rounded (no contraction), so that every kernel and every column of a
// grid evaluates the same sequence of roundings; those of the WENO functions are left to the compiler.
#pragma once

#include "vlb_internal.cuh"

namespace vlb {

template <typename V> struct LaneOf { using S = V; };
template <> struct LaneOf<float2> { using S = float; };

__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

template <typename V>
__device__ __forceinline__ V bc(typename LaneOf<V>::S x) {
  if constexpr (sizeof(V) == 8 && sizeof(typename LaneOf<V>::S) == 4)
    return make_float2(x, x);
  else
    return x;
}

__device__ __forceinline__ float node_recip(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double node_recip(double x) { return __drcp_rn(x); }

// Velocity constants in the parity basis (index 0: b, 1: a): kap maps even to odd, lam odd to even
// (both with the basis's normalisation 1/4 folded in), ww = w_x w_y.
// fix: 1 - sum w v v with the constants as they are rounded (FP32: -4.0e-8, nearly all from a, which rounds up by a
// third of an ulp).
template <typename T>
struct alignas(16) NodeConst {  // 16-byte loads of what follows it in a kernel's parameters
  T v[2], v2[2], kap[2][2], lam[2][2], ww[2][2], fix;
};

template <typename T>
NodeConst<T> make_node_const() {
  const VelocityConsts d = velocity_consts();
  const int pos[2] = {3, 2}, neg[2] = {0, 1};
  NodeConst<T> c;
  for (int x = 0; x < 2; ++x) {
    c.v[x] = (T)d.v[pos[x]];
    c.v2[x] = (T)(d.v[pos[x]] * d.v[pos[x]]);
    for (int y = 0; y < 2; ++y) {
      c.kap[x][y] = (T)(0.25 * (d.K[pos[x]][pos[y]] + d.K[pos[x]][neg[y]]));
      c.lam[x][y] = (T)(0.25 * (d.K[pos[x]][pos[y]] - d.K[pos[x]][neg[y]]));
      c.ww[x][y] = (T)(d.w[pos[x]] * d.w[pos[y]]);
    }
  }
  double m2 = 0.0;
  for (int x = 0; x < 2; ++x)
    for (int y = 0; y < 2; ++y) m2 += 4.0 * c.ww[x][y] * c.v[x] * c.v[x];
  c.fix = (T)(1.0 - m2);
  return c;
}

// Velocity m inv of the equilibrium, FP32: times 1 + fix, in one rounding.  Without it the momentum of the equilibrium is
// 1 + 4.0e-8 times that of the populations, the same at every node, and the momentum grows by 4.0e-8 dt / tau in
// every stage: 1e-6 of it after 64 steps at dt / tau = 0.6, more than all other roundings together.
template <typename V, typename T>
__device__ __forceinline__ V node_velocity(V m, V inv, T fix) {
  if constexpr (sizeof(T) == 4) return vfma(m, inv, vmul(vmul(bc<V>(fix), m), inv));
  return vmul(m, inv);
}

// Row table: everything of the right-hand side that depends on the theta row alone, times dt (about 70
// operations that every node would otherwise repeat).  Entry e of row q is
//   S (c1 X1(q) Y + c2 X2(q))  -  [e >= E_CC] dt / tau
// with X1, X2 coefficient arrays, S one of dt, M dt, kappa and 1, and Y one of 1, J(q - 2 .. q + 2).
// FP32 pair kernels read the 32-entry rows of a table in global memory, formed once per handle in FP64
// (row_table_entry rounds it); the FP64 direct kernel forms the rows of its tile in shared memory.
enum RowEntry : int {
  E_GBB = 0,  // Gamma v_b^2, Gamma v_b v_a, Gamma v_a^2
  E_GBA,
  E_GAA,
  E_EM,   // (E_pos + E_neg) / 2 of the rest-state residual
  E_NEB,  // v_x (E_pos - E_neg) / 2, x = b, a
  E_NEA,
  E_GP,   // 1 / (2 R J dvarphi)
  E_LP,   // M times the Laplace-Beltrami coefficients: varphi, theta
  E_LT,
  E_XN,   // Cahn-Hilliard advection: J(q + 1), J(q - 1) over 2 r J dtheta; 1 / (2 R J dvarphi)
  E_XS,
  E_YP,
  E_JP,   // J(q + 1/2), J(q - 1/2) (not folded into E_LT, E_KT: neighbouring rows share the rounded value)
  E_JM,
  E_KT,   // kappa times the Laplace-Beltrami coefficients (for mu; not times dt): theta, varphi
  E_KP,
  E_TH,   // per x, 8 entries: theta taps of -v (flux difference) (RowTap), then v_x / (6 R J dvarphi)
  E_PV6 = E_TH + 16,  // FP64: 6 and -2 times the varphi weight, then the sum of the centre taps per (x, y)
  E_PV2 = E_PV6 + 2,
  E_CC = E_PV2 + 2,
  NROW32 = E_PV6,
  NROW64 = E_CC + 4
};
enum RowTap : int { TAP_FARP = 0, TAP_NEARP, TAP_DOWNN, TAP_MID, TAP_NEARN, TAP_DOWNP, TAP_FARN, TAP_PV };
template <typename T>
constexpr int row_entries() { return sizeof(T) == 8 ? NROW64 : NROW32; }

// One entry's rule; y: 0 none, 1 .. 5 J(q - 2) .. J(q + 2); s: 0 dt, 1 M dt,
// 2 kappa, 3 one.
// Compile-time tables in global memory: lanes of a warp read different entries, which a constant bank serialises.
template <typename T>
struct RowRule {
  T c1, c2;
  unsigned char s, x1, y, x2;
};
template <typename T>
struct RowRules {
  RowRule<T> e[NROW64];
};
constexpr double csqrt(double x) {
  double r = x;
  for (int i = 0; i < 60; ++i) r = 0.5 * (r + x / r);
  return r;
}
constexpr double kVelA = csqrt(3.0 - csqrt(6.0)), kVelB = csqrt(3.0 + csqrt(6.0));  // Eq. vmatrix

template <typename T>
constexpr RowRules<T> make_row_rules() {
  RowRules<T> r{};
  auto set = [&](int e, double c1, int s, int x1, int y, double c2 = 0.0, int x2 = 0) {
    r.e[e] = RowRule<T>{(T)c1, (T)c2, (unsigned char)s, (unsigned char)x1, (unsigned char)y, (unsigned char)x2};
  };
  const double v[2] = {kVelB, kVelA};
  set(E_GBB, v[0] * v[0], 0, C_GAM, 0);
  set(E_GBA, v[0] * v[1], 0, C_GAM, 0);
  set(E_GAA, v[1] * v[1], 0, C_GAM, 0);
  set(E_EM, 0.5, 0, C_EP, 0, 0.5, C_EN);
  set(E_GP, 1.0, 0, C_GP, 0);
  set(E_LP, 1.0, 1, C_LP, 0);
  set(E_LT, 1.0, 1, C_LT, 0);
  set(E_JP, 1.0, 3, C_JP, 0);
  set(E_JM, 1.0, 3, C_JM, 0);
  set(E_KT, 1.0, 2, C_LT, 0);
  set(E_KP, 1.0, 2, C_LP, 0);
  set(E_XN, 0.5, 0, C_CT, 4);
  set(E_XS, 0.5, 0, C_CT, 2);
  set(E_YP, 0.5, 0, C_CP, 0);
  for (int x = 0; x < 2; ++x) {
    set(E_NEB + x, 0.5 * v[x], 0, C_EP, 0, -0.5 * v[x], C_EN);
    const int t = E_TH + 8 * x;
    set(t + TAP_PV, v[x] / 6.0, 0, C_CP, 0);
    set(t + TAP_FARP, -v[x] / 6.0, 0, C_CT, 1);
    set(t + TAP_NEARP, v[x], 0, C_CT, 2);
    set(t + TAP_DOWNN, -v[x] / 3.0, 0, C_CT, 2);
    set(t + TAP_MID, -v[x] / 2.0, 0, C_CT, 3);
    set(t + TAP_NEARN, v[x], 0, C_CT, 4);
    set(t + TAP_DOWNP, -v[x] / 3.0, 0, C_CT, 4);
    set(t + TAP_FARN, -v[x] / 6.0, 0, C_CT, 5);
    set(E_PV6 + x, v[x], 0, C_CP, 0);
    set(E_PV2 + x, -v[x] / 3.0, 0, C_CP, 0);
    for (int y = 0; y < 2; ++y) set(E_CC + 2 * x + y, -v[x] / 2.0, 0, C_CT, 3, -v[y] / 2.0, C_CP);
  }
  return r;
}

// Entry of row q by rule r (a lane each), or (row_entry<e>) for an entry known at compile time.
template <typename T>
__device__ __forceinline__ T row_entry(const RowRule<T>& r, const StageArgs<T>& a, int q, bool centre) {
  const int nt = a.nt, y = r.y, s = r.s;
  const T sc = s == 3 ? T(1) : (s == 2 ? a.kappa : (s == 1 ? vmul(a.dt, a.M) : a.dt));
  T v = vmul(vmul(r.c1, sc), a.coef[(int64_t)r.x1 * nt + q]);
  if (y) {
    int row = q + y - 3;
    row += row < 0 ? nt : (row >= nt ? -nt : 0);
    v = vmul(v, a.coef[(int64_t)C_J * nt + row]);
  }
  if (r.c2 != T(0)) v = vfma(vmul(r.c2, sc), a.coef[(int64_t)r.x2 * nt + q], v);
  if (centre) v = vfma(-a.dt, a.inv_tau, v);
  return v;
}
template <typename T>
__device__ __forceinline__ void row_all(T (&rt)[row_entries<T>()], const StageArgs<T>& a, int q) {
  constexpr RowRules<T> R = make_row_rules<T>();
#pragma unroll
  for (int e = 0; e < row_entries<T>(); ++e) rt[e] = row_entry(R.e[e], a, q, e >= E_CC);
}

// Entry k of the FP32 row table from its FP64 value v, lane k of a whole warp holding entry k of the row.  The four theta
// taps of a velocity nearly cancel, and what their roundings leave of the sum acts on the population itself, the same
// in every stage; so the smallest of them, the far tap, is rounded to the sum less the other three as they are
// rounded.  176 x 32 at tau = 0.1, 10 steps: error of the populations 1.09e-7 with four taps rounded for themselves.
__device__ __forceinline__ float row_table_entry(double v, int k) {
  const float own = (float)v;
  const int t = k & 7, th = k - t;  // E_TH is a multiple of 8
  const bool far = k >= E_TH && (t == TAP_FARP || t == TAP_FARN);
  const int near = far ? th + (t == TAP_FARP ? TAP_NEARP : TAP_NEARN) : k;
  const int down = far ? th + (t == TAP_FARP ? TAP_DOWNP : TAP_DOWNN) : k, mid = far ? th + TAP_MID : k;
  const double sum = v + __shfl_sync(0xffffffffu, v, near) + __shfl_sync(0xffffffffu, v, mid) +
                     __shfl_sync(0xffffffffu, v, down);
  const double rest = (double)__shfl_sync(0xffffffffu, own, near) + __shfl_sync(0xffffffffu, own, mid) +
                      __shfl_sync(0xffffffffu, own, down);
  return far ? (float)(sum - rest) : own;
}

// (x_0 .. x_3) at velocities (-b, -a, a, b) <-> (E_b, E_a, O_b, O_a)
template <typename V>
__device__ __forceinline__ void to_parity(V& x0, V& x1, V& x2, V& x3) {
  const V eb = vadd(x3, x0), ea = vadd(x2, x1), ob = vsub(x3, x0), oa = vsub(x2, x1);
  x0 = eb;
  x1 = ea;
  x2 = ob;
  x3 = oa;
}
template <typename V>
__device__ __forceinline__ void from_parity(V& x0, V& x1, V& x2, V& x3) {
  const V pb = vadd(x0, x2), mb = vsub(x0, x2), pa = vadd(x1, x3), ma = vsub(x1, x3);
  x0 = mb;
  x1 = ma;
  x2 = pa;
  x3 = pb;
}

// g[4 i + j] (i: theta velocity, j: varphi velocity) -> P[4 ci + cj]
template <typename V>
__device__ __forceinline__ void to_parity16(V (&g)[16]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) to_parity(g[4 * i], g[4 * i + 1], g[4 * i + 2], g[4 * i + 3]);
#pragma unroll
  for (int j = 0; j < 4; ++j) to_parity(g[j], g[4 + j], g[8 + j], g[12 + j]);
}
template <typename V>
__device__ __forceinline__ void from_parity16(V (&r)[16]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) from_parity(r[j], r[4 + j], r[8 + j], r[12 + j]);
#pragma unroll
  for (int i = 0; i < 4; ++i) from_parity(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
}

// Deviation of the density and the momentum density (Sec. 2.3) from the parity combinations.
template <typename V, typename T>
__device__ __forceinline__ void parity_moments(const V (&P)[16], const NodeConst<T>& nc, V& dn, V& mt, V& mp) {
  dn = vadd(vadd(P[0], P[1]), vadd(P[4], P[5]));
  mt = vfma(bc<V>(nc.v[0]), vadd(P[8], P[9]), vmul(bc<V>(nc.v[1]), vadd(P[12], P[13])));
  mp = vfma(bc<V>(nc.v[0]), vadd(P[2], P[6]), vmul(bc<V>(nc.v[1]), vadd(P[3], P[7])));
}

// Velocity-space terms of the right-hand side times dt, from the combinations P:
//   dt { (Gamma v_j^2 - F^theta) K g  +  K~-term (-F^phi - Gamma v_i v_j)  +  w_i w_j X },
//   X = (dn + n (poly - 1)) / tau + n0 v_i (E(sign v_i) + F^theta) + n0 v_j F^phi
// (poly the third-order Hermite polynomial of Eq. feq; the -g/tau part is left to the caller), turned
// back to populations in R.  Ft, Fp and itau arrive multiplied by dt; rt is the node's row of the table.
template <typename V, typename T>
__device__ __forceinline__ void velocity_space(const V (&P)[16], V (&R)[16], const NodeConst<T>& nc, const T* rt, V Ft,
                                               V Fp, T itau, T n0, V dn, V ut, V up) {
  const V g[2][2] = {{bc<V>(rt[E_GBB]), bc<V>(rt[E_GBA])}, {bc<V>(rt[E_GBA]), bc<V>(rt[E_GAA])}};
#pragma unroll
  for (int cj = 0; cj < 4; ++cj) {  // (Gamma v_j^2 - F^theta) K along theta velocities
    const V c = vsub(g[cj & 1][cj & 1], Ft);
    const V q0 = vmul(c, P[cj]), q1 = vmul(c, P[4 + cj]), q2 = vmul(c, P[8 + cj]), q3 = vmul(c, P[12 + cj]);
    R[8 + cj] = vfma(bc<V>(nc.kap[0][1]), q1, vmul(bc<V>(nc.kap[0][0]), q0));
    R[12 + cj] = vfma(bc<V>(nc.kap[1][1]), q1, vmul(bc<V>(nc.kap[1][0]), q0));
    R[cj] = vfma(bc<V>(nc.lam[0][1]), q3, vmul(bc<V>(nc.lam[0][0]), q2));
    R[4 + cj] = vfma(bc<V>(nc.lam[1][1]), q3, vmul(bc<V>(nc.lam[1][0]), q2));
  }
#pragma unroll
  for (int ci = 0; ci < 4; ++ci) {
    // minus K along varphi velocities of (F^phi + Gamma v_i v_m) g: v_i v_m flips both parities
    const int x = ci & 1, cb = 4 * (ci ^ 2), c0 = 4 * ci;
    const V h0 = vfma(g[x][0], P[cb + 2], vmul(Fp, P[c0])), h1 = vfma(g[x][1], P[cb + 3], vmul(Fp, P[c0 + 1]));
    const V h2 = vfma(g[x][0], P[cb], vmul(Fp, P[c0 + 2])), h3 = vfma(g[x][1], P[cb + 1], vmul(Fp, P[c0 + 3]));
    R[c0 + 2] = vfma(bc<V>(-nc.kap[0][0]), h0, vfma(bc<V>(-nc.kap[0][1]), h1, R[c0 + 2]));
    R[c0 + 3] = vfma(bc<V>(-nc.kap[1][0]), h0, vfma(bc<V>(-nc.kap[1][1]), h1, R[c0 + 3]));
    R[c0] = vfma(bc<V>(-nc.lam[0][0]), h2, vfma(bc<V>(-nc.lam[0][1]), h3, R[c0]));
    R[c0 + 1] = vfma(bc<V>(-nc.lam[1][0]), h2, vfma(bc<V>(-nc.lam[1][1]), h3, R[c0 + 1]));
  }
  // equilibrium and reference part, with A = v_x u^theta, B = v_y u^phi per velocity magnitude
  const V dntau = vmul(dn, bc<V>(itau)), ntau = vfma(bc<V>(itau), bc<V>(n0), dntau);
  const V hut = vmul(vmul(bc<V>(T(0.5)), ut), ut), hup = vmul(vmul(bc<V>(T(0.5)), up), up);
  const V us = vadd(hut, hup), one = vsub(bc<V>(T(1)), us);
  const V tF = vmul(bc<V>(n0), vadd(Ft, bc<V>(rt[E_EM]))), pF = vmul(bc<V>(n0), Fp);
  const V nut = vmul(ntau, ut), nup = vmul(ntau, up);
  const V third = bc<V>(T(1) / T(3));
  V hB[2], B[2], nhB[2], nB[2], pB[2];
#pragma unroll
  for (int y = 0; y < 2; ++y) {
    hB[y] = vmul(bc<V>(nc.v2[y]), hup);
    B[y] = vmul(bc<V>(nc.v[y]), up);
    nhB[y] = vmul(ntau, hB[y]);
    nB[y] = vmul(bc<V>(nc.v[y]), nup);
    pB[y] = vmul(bc<V>(nc.v[y]), pF);
  }
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const V hA = vmul(bc<V>(nc.v2[x]), hut), nA = vmul(bc<V>(nc.v[x]), nut);
    const V pre = vfma(ntau, vsub(hA, us), vfma(bc<V>(n0), bc<V>(rt[E_NEB + x]), dntau));
    const V cx = vfma(third, hA, one), dx = vmul(bc<V>(nc.v[x]), tF), ox = vadd(hA, one);
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      const V w = bc<V>(nc.ww[x][y]);
      R[4 * x + y] = vfma(w, vadd(pre, nhB[y]), R[4 * x + y]);
      R[4 * x + 8 + y] = vfma(w, vfma(nA, vadd(cx, hB[y]), dx), R[4 * x + 8 + y]);
      R[4 * x + y + 2] = vfma(w, vfma(nB[y], vfma(third, hB[y], ox), pB[y]), R[4 * x + y + 2]);
      R[4 * x + 8 + y + 2] = vfma(w, vmul(nA, B[y]), R[4 * x + 8 + y + 2]);
    }
  }
  from_parity16(R);
}

// Fifth-order WENO-JS face value between g2 and g3 of the window g0..g4, upwind from g0's side.
template <typename T>
__device__ __forceinline__ T weno5(T g0, T g1, T g2, T g3, T g4) {
  const T c13_12 = T(13) / T(12), sixth = T(1) / T(6), eps = T(1e-6);
  T q0 = (T(2) * g0 - T(7) * g1 + T(11) * g2) * sixth;
  T q1 = (-g1 + T(5) * g2 + T(2) * g3) * sixth;
  T q2 = (T(2) * g2 + T(5) * g3 - g4) * sixth;
  T d0 = g0 - T(2) * g1 + g2, e0 = g0 - T(4) * g1 + T(3) * g2;
  T d1 = g1 - T(2) * g2 + g3, e1 = g1 - g3;
  T d2 = g2 - T(2) * g3 + g4, e2 = T(3) * g2 - T(4) * g3 + g4;
  T b0 = c13_12 * d0 * d0 + T(0.25) * e0 * e0;
  T b1 = c13_12 * d1 * d1 + T(0.25) * e1 * e1;
  T b2 = c13_12 * d2 * d2 + T(0.25) * e2 * e2;
  T a0 = T(0.1) / ((eps + b0) * (eps + b0));
  T a1 = T(0.6) / ((eps + b1) * (eps + b1));
  T a2 = T(0.3) / ((eps + b2) * (eps + b2));
  return (a0 * q0 + a1 * q1 + a2 * q2) / (a0 + a1 + a2);
}

// a / b with b in the range of the weights: FP32 within 2 ulp (it scales a correction to g2)
__device__ __forceinline__ float quotient(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double quotient(double a, double b) { return a * node_recip(b); }

// The same face value with one reciprocal instead of four divisions: the weights d_k / s_k^2 times (s_0 s_1 s_2)^2.
// Sets `bad` where the weights leave the range in which no product overflows (differences of about 3000 in
// FP32, or a value that is not finite): the caller then takes weno5.
template <typename T>
__device__ __forceinline__ T weno5_face(T g0, T g1, T g2, T g3, T g4, bool& bad) {
  const T c = T(13) / T(12), eps = T(1e-6);
  const T f1 = g1 - g0, f2 = g2 - g1, f3 = g3 - g2, f4 = g4 - g3;
  const T d0 = f2 - f1, d1 = f3 - f2, d2 = f4 - f3;
  const T e0 = d0 + T(2) * f2, e1 = f2 + f3, e2 = d2 - T(2) * f3;  // g0 - 4 g1 + 3 g2, g3 - g1, 3 g2 - 4 g3 + g4
  const T s0 = (c * d0) * d0 + ((T(0.25) * e0) * e0 + eps), s1 = (c * d1) * d1 + ((T(0.25) * e1) * e1 + eps);
  const T s2 = (c * d2) * d2 + ((T(0.25) * e2) * e2 + eps);
  const T p0 = s1 * s2, p1 = s0 * s2, p2 = s0 * s1;
  const T w0 = (T(0.1) * p0) * p0, w1 = (T(0.6) * p1) * p1, w2 = (T(0.3) * p2) * p2, w = w0 + w1 + w2;
  bad = bad || !(w <= (sizeof(T) == 4 ? T(1e30) : T(1e250)));
  // face values relative to g2: (5 f2 - 2 f1) / 6, (f2 + 2 f3) / 6, (4 f3 - f4) / 6
  const T num = w0 * (T(5) * f2 - T(2) * f1) + w1 * (f2 + T(2) * f3) + w2 * (T(4) * f3 - f4);
  return g2 + quotient(num, w * T(6));
}

// WENO5 flux difference face_{+1/2} - face_{-1/2} at the centre x[3] of a 7-point window.
template <typename T, bool POS>
__device__ __forceinline__ T weno_diff(const T (&x)[7]) {
  if (POS) return weno5(x[1], x[2], x[3], x[4], x[5]) - weno5(x[0], x[1], x[2], x[3], x[4]);
  return weno5(x[6], x[5], x[4], x[3], x[2]) - weno5(x[5], x[4], x[3], x[2], x[1]);
}

}  // namespace vlb
