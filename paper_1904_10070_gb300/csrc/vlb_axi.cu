// Axisymmetric special case, n_phi = 1.  With one varphi column every varphi difference is zero:
// the varphi flux of f and of u^phi phi, the varphi part of the Laplace-Beltrami operator and the
// force component F^phi all vanish, while u^phi itself (a swirl) and the inertial terms through
// Gamma and K~ remain.
//
// One thread-block cluster holds the column: CTA c owns a block of consecutive rows, keeps the three
// Runge-Kutta states of its rows and of H halo rows on each side in shared memory (UW3: H = 2, WENO5: 3),
// and runs `steps` whole steps.  Per stage: four threads a row (thread i: theta velocity v_i) form the
// moments and mu of the owned rows and one row on each side; after a CTA barrier they evaluate the
// right-hand sides and the update, write the new rows to the next state's buffer and push the boundary rows
// into the two neighbours' halos with asynchronous stores that complete on the neighbour's mbarrier (one per
// side and parity of the stage: a neighbour can run at most one stage ahead, since its next stage needs this
// CTA's push).  Nothing but the first and the last state touches global memory.  Every wait is bounded; one
// that gives up raises the handle's flag (2).
// The kernels are bound by the latency of that chain, FP64 by the SMs' FP64 units.  A cluster barrier per
// stage instead of the counted pushes cost 0.6 us a stage (its release fence waits for the remote stores).
// Per step: 320 rows FP32 8.5 us for the single CTA over L1 / L2 that this replaces, 4.0 with 16 CTAs and
// cluster barriers, 2.1 with pushes (axi16_kernel); FP64 240 us (512 rows) -> 22 us (320 rows).
#include <algorithm>

#include "vlb_node.cuh"

namespace vlb {

namespace {

constexpr int kAxiCta = 16, kAxiPortable = 8;  // CTAs per cluster: with the non-portable opt-in, without
constexpr int kRowVals = 33;                    // per-row values kept in shared memory, at most (AxiRow, or the row table)
constexpr int kAxiThreads = 256;

template <typename T>
struct AxiConst {
  T v[4], K[4][4], ww[4][4], fix;  // fix: of node_velocity
};

// everything a row needs, times dt where it multiplies a rate
template <typename T>
struct AxiRow {
  T w[5];         // dt J(q - 2 .. q + 2) / (6 r J dtheta)
  T gam, em, ed;  // dt Gamma, dt (E_pos + E_neg) / 2, dt (E_pos - E_neg) / 2
  T lt, kt;       // dt M and kappa times the Laplace-Beltrami coefficient
  T jp, jm;       // J(q +- 1/2)
  T xn, xs;       // dt J(q +- 1) / (2 r J dtheta)
  T ct;           // dt / (r J dtheta)
};
static_assert(sizeof(AxiRow<float>) <= kRowVals * sizeof(float), "one array entry per value");

__device__ __forceinline__ int axi_wrap(int x, int n) {
  x %= n;
  return x < 0 ? x + n : x;
}

template <typename T>
__device__ __forceinline__ AxiRow<T> axi_row(const StageArgs<T>& a, int q) {
  const int nt = a.nt;
  auto C = [&](int k, int row) { return a.coef[(int64_t)k * nt + axi_wrap(row, nt)]; };
  AxiRow<T> r;
  const T ct = C(C_CT, q) * a.dt, lt = C(C_LT, q), ep = C(C_EP, q) * a.dt, en = C(C_EN, q) * a.dt;
  r.ct = ct;
#pragma unroll
  for (int d = 0; d < 5; ++d) r.w[d] = ct * C(C_J, q + d - 2) * T(1.0 / 6.0);
  r.gam = C(C_GAM, q) * a.dt;
  r.em = T(0.5) * (ep + en);
  r.ed = T(0.5) * (ep - en);
  r.jp = C(C_JP, q);
  r.jm = C(C_JM, q);
  r.lt = a.dt * a.M * lt;
  r.kt = a.kappa * lt;
  r.xn = T(0.5) * ct * C(C_J, q + 1);
  r.xs = T(0.5) * ct * C(C_J, q - 1);
  return r;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t remote_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

__device__ __forceinline__ void mbar_init1(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
// acquire at cluster scope: the neighbours' pushes are visible after it; bounded
__device__ __forceinline__ bool mbar_wait1(uint64_t* bar, uint32_t parity) {
  for (int it = 0; it < (1 << 22); ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, "
        "p;\n}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}
// asynchronous store into a CTA of the cluster, counted on that CTA's barrier
__device__ __forceinline__ void push(uint32_t addr, float v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];\n" ::"r"(addr), "f"(v), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void push(uint32_t addr, double v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];\n" ::"r"(addr), "d"(v), "r"(bar)
               : "memory");
}

// rows of CTA c of nc: the first nt % nc CTAs own one row more
__host__ __device__ constexpr int axi_first(int nt, int nc, int c) {
  return c * (nt / nc) + (c < nt % nc ? c : nt % nc);
}
__host__ __device__ constexpr int axi_count(int nt, int nc, int c) { return nt / nc + (c < nt % nc ? 1 : 0); }

constexpr size_t kSmemMax = 232448;  // opt-in shared memory of one CTA

// pitch of one array of a state buffer: the rows and their halos, padded so that the four velocity rows
// of a warp (4 pitch apart) fall on different banks, unless the padding is what does not fit (the longest FP64
// columns on eight CTAs)
template <typename T>
__host__ __device__ constexpr int axi_pitch(int rows, int H) {
  int p = rows + 2 * H;
  while (p % 8 != 2) ++p;
  return 32 + sizeof(T) * ((size_t)3 * state_arrays(sizeof(T)) * p + 5 * (size_t)(rows + 2)) <= kSmemMax ? p : rows + 2 * H;
}

// FP32 UW3 columns read the handle's row table; the others form an AxiRow from the coefficient arrays
template <typename T, int ADV>
__host__ __device__ constexpr bool row_table() { return sizeof(T) == 4 && ADV == VLB_UW3; }

template <typename T, int ADV>
constexpr size_t axi_smem(int nt, int nc, bool table) {
  const int rmax = axi_count(nt, nc, 0), H = ADV == VLB_UW3 ? 2 : 3;
  const size_t elems = (size_t)3 * state_arrays(sizeof(T)) * axi_pitch<T>(rmax, H) + 5 * (size_t)(rmax + 2) +
                       (table ? (size_t)(rmax + 2) * (row_table<T, ADV>() ? kRowVals : sizeof(AxiRow<T>) / sizeof(T)) : 0);
  return 32 + elems * sizeof(T);
}
static_assert(axi_smem<double, VLB_UW3>(kAxiMaxRows, kAxiPortable, false) <= kSmemMax &&
                  axi_smem<double, VLB_WENO5>(kAxiMaxRows, kAxiPortable, false) <= kSmemMax &&
                  axi_smem<float, VLB_UW3>(kAxiMaxRows, kAxiPortable, true) <= kSmemMax &&
                  axi_smem<float, VLB_WENO5>(kAxiMaxRows, kAxiPortable, false) <= kSmemMax,
              "every column fits a cluster of the portable size");

// `steps` SSP-RK3 steps in the Shu-Osher form of run_steps: U1 = U + dt L(U); U2 = U + 1/4 (U1 - U + dt L(U1));
// U <- U + 2/3 (U2 - U + dt L(U2)).  The third stage writes U in place: a thread reads its own U before it
// overwrites it, and nobody reads U's halo rows in that stage, so the neighbours may already push the new ones.
template <typename T, int ADV, int CH>
__global__ void __launch_bounds__(kAxiThreads) axi_kernel(StageArgs<T> a, const __grid_constant__ AxiConst<T> ac, T* U,
                                                          int steps, int table) {
  constexpr bool DF = sizeof(T) == 4;  // phi as a float pair in FP32 storage
  constexpr int H = ADV == VLB_UW3 ? 2 : 3, NST = DF ? NARR + 1 : NARR;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nt = a.nt, nc = gridDim.x, c = blockIdx.x, tid = threadIdx.x;  // one cluster: rank = blockIdx.x
  const int r0 = axi_first(nt, nc, c), R = axi_count(nt, nc, c), rmax = axi_count(nt, nc, 0);
  const int P = axi_pitch<T>(rmax, H), SZ = NST * P;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);  // [from prev, from next][parity of the stage]
  T* buf = reinterpret_cast<T*>(smem_raw + 32);  // three states, array k of state s at buf + s SZ + k P, row r at H + r
  T *s_dn = buf + 3 * SZ, *s_in = s_dn + rmax + 2, *s_ut = s_in + rmax + 2, *s_up = s_ut + rmax + 2;
  T* s_mu = s_up + rmax + 2;
  constexpr bool RT = row_table<T, ADV>();
  AxiRow<T>* s_row = reinterpret_cast<AxiRow<T>*>(s_mu + rmax + 2);  // rows -1 .. R
  T* s_rt = s_mu + rmax + 2;                                          // or, with the row table, 33 a row
  for (int k = 0; k < NST; ++k)
    for (int r = tid; r < R + 2 * H; r += kAxiThreads)
      buf[k * P + r] = U[k * a.stride + axi_wrap(r0 + r - H, nt)];
  if constexpr (RT) {  // always fits (host)
    for (int x = tid; x < (R + 2) * kRowTable; x += kAxiThreads)
      s_rt[x / kRowTable * 33 + x % kRowTable] =
          a.rows[(int64_t)axi_wrap(r0 + x / kRowTable - 1, nt) * kRowTable + x % kRowTable];
  } else if (table) {
    for (int r = tid; r < R + 2; r += kAxiThreads) s_row[r] = axi_row(a, axi_wrap(r0 + r - 1, nt));
  }
  // the neighbours' halo slots of this CTA's first and last H rows
  const int cp = c > 0 ? c - 1 : nc - 1, cn = c + 1 < nc ? c + 1 : 0;
  const uint32_t base = smem_addr(buf), to_prev = remote_addr(base, cp), to_next = remote_addr(base, cn);
  const int shift_prev = axi_count(nt, nc, cp), shift_next = -R;  // row r of this CTA as the neighbour's row
  const uint32_t bar_prev = remote_addr(smem_addr(bar + 2), cp), bar_next = remote_addr(smem_addr(bar), cn);
  if (tid == 0) {
    for (int x = 0; x < 4; ++x) mbar_init1(bar + x);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  cluster_barrier();
  uint32_t stage = 0;
  bool ok = true;

  const int i = tid & 3;  // this thread's theta velocity
  const bool pos = i >= 2;
  const T vi = ac.v[i], K0 = ac.K[i][0], K1 = ac.K[i][1], K2 = ac.K[i][2], K3 = ac.K[i][3];
  const T itau = a.inv_tau * a.dt, av = pos ? vi : -vi;
  const T ivb = T(1) / ac.v[3], iva = T(1) / ac.v[2];
  for (int n = 0; n < steps && ok; ++n) {
#pragma unroll 1
    for (int st = 0; st < 3; ++st, ++stage) {
      const uint32_t par = stage & 1, phase = (stage >> 1) & 1;
      if (tid == 0) {  // armed before this CTA's own pushes, which let the neighbours run one stage ahead
        mbar_expect(bar + par, H * NST * sizeof(T));
        mbar_expect(bar + 2 + par, H * NST * sizeof(T));
      }
      const T* in = buf + st * SZ;
      const int ob = st == 2 ? 0 : st + 1;  // output buffer
      T* out = buf + ob * SZ;
      const T b = st == 0 ? T(1) : (st == 1 ? T(0.25) : T(2.0 / 3.0));
      // moments (Sec. 2.3) and mu (Eq. mu) of rows -1 .. R
      for (int it = tid; it < ((R + 2) * 4 + 31) / 32 * 32; it += kAxiThreads) {
        const int row = min(it >> 2, R + 1);  // surplus lanes repeat the last row (whole warps shuffle)
        const T* f = in + 4 * i * P + H + row - 1;
        const T g0 = f[0], g1 = f[P], g2 = f[2 * P], g3 = f[3 * P];
        // sums over j, then over i in the opposite pairs (differences first: v_1 = -v_4, v_2 = -v_3)
        T dn = (g0 + g3) + (g1 + g2);
        T mp = ac.v[3] * (g3 - g0) + ac.v[2] * (g2 - g1);
        const T dx = __shfl_xor_sync(0xffffffffu, dn, 3);
        T mt = av * (pos ? dn - dx : dx - dn);
        dn += dx;
        mp += __shfl_xor_sync(0xffffffffu, mp, 3);
        dn += __shfl_xor_sync(0xffffffffu, dn, 1);
        mt += __shfl_xor_sync(0xffffffffu, mt, 1);
        mp += __shfl_xor_sync(0xffffffffu, mp, 1);
        const T* ph = in + NPOP * P + H + row - 1;
        const T p0 = ph[0];
        T dN = ph[1] - p0, dS = p0 - ph[-1], lo = T(0);
        if (DF) {
          const T* pl = ph + P;
          lo = pl[0];
          dN += pl[1] - lo;
          dS += lo - pl[-1];
        }
        T kt, jp, jm;
        if constexpr (RT) {
          kt = s_rt[row * 33 + E_KT];
          jp = s_rt[row * 33 + E_JP];
          jm = s_rt[row * 33 + E_JM];
        } else {
          const AxiRow<T> rv = table ? s_row[row] : axi_row(a, axi_wrap(r0 + row - 1, nt));
          kt = rv.kt;
          jp = rv.jp;
          jm = rv.jm;
        }
        if (i == 0 && (it >> 2) <= R + 1) {
          const T inv_n = node_recip(vadd(a.n0, dn));
          const T cubic = p0 * (T(1) - p0 * p0) + (T(1) - T(3) * p0 * p0) * lo;  // at hi + lo, first order in lo
          s_dn[row] = dn;
          s_in[row] = inv_n;
          s_ut[row] = node_velocity(mt, inv_n, ac.fix);
          s_up[row] = node_velocity(mp, inv_n, ac.fix);
          s_mu[row] = -a.A * cubic - kt * (jp * dN - jm * dS);
        }
      }
      __syncthreads();
      for (int it = tid; it < R * 4; it += kAxiThreads) {
        const int row = it >> 2, m = row + 1;
        AxiRow<T> rv = {};
        const T* rt = s_rt + m * 33;
        if constexpr (!RT) rv = table ? s_row[m] : axi_row(a, r0 + row);
        const T dn = s_dn[m], ut = s_ut[m], up = s_up[m], mu_c = s_mu[m], mu_n = s_mu[m + 1], mu_s = s_mu[m - 1];
        const T* ph = in + NPOP * P + H + row;
        const T* u0 = buf + H + row;
        T o[6];
        int nout = 4, k0 = 4 * i;
        T Ft = T(0);
        if (CH == VLB_HYDRO) Ft = ph[0] * s_in[m] * (mu_s - mu_n) * (a.gt * a.dt);  // Eq. pbin
        T g[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) g[k] = in[k * P + H + row];
        // n / tau from the density that was inverted for u: n0 / tau rounded on its own would be off by the same amount
        // at every node and stage, and the momentum would drift by it
        const T usq = ut * ut + up * up, c0 = T(1) - T(0.5) * usq, hu = T(-0.5) * usq;
        const T dntau = vmul(dn, itau), ntau = vmul(vadd(a.n0, dn), itau), ai = vmul(vi, ut);
        const bool big = i == 0 || i == 3;
        const T em = RT ? rt[E_EM] : rv.em, ne = RT ? (big ? rt[E_NEB] : rt[E_NEA]) : av * rv.ed;
        const T ci = dntau + a.n0 * (vi * (em + Ft) + ne);
        // Gamma v_j^2 and Gamma v_i v_m by magnitude
        const T gb2 = RT ? rt[E_GBB] : rv.gam * ac.v[3] * ac.v[3], ga2 = RT ? rt[E_GAA] : rv.gam * ac.v[2] * ac.v[2];
        const T gab = RT ? rt[E_GBA] : rv.gam * ac.v[3] * ac.v[2];
        T hb = big ? gb2 : gab, ha = big ? gab : ga2;
        hb = pos ? hb : -hb;
        ha = pos ? ha : -ha;
        T tf, tn, tm, td;
        if constexpr (RT) {  // tm: the sum of the four taps, v_i (E + Gamma)
          const T* t = rt + E_TH + (big ? 0 : 8);
          tf = t[pos ? TAP_FARP : TAP_FARN];
          tn = t[pos ? TAP_NEARP : TAP_NEARN];
          td = t[pos ? TAP_DOWNP : TAP_DOWNN];
          const T gv = big ? gb2 * ivb : ga2 * iva;
          tm = vadd(vfma(vi, em, ne), pos ? gv : -gv);
        } else {
          tf = -av * (pos ? rv.w[0] : rv.w[4]);
          tn = T(6) * av * (pos ? rv.w[1] : rv.w[3]);
          tm = T(-3) * av * rv.w[2];
          td = T(-2) * av * (pos ? rv.w[3] : rv.w[1]);
        }
        const T* fi = in + 4 * i * P + H + row;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const T* fk = fi + j * P;
          const T gk = fk[0];
          T acc;
          if (ADV == VLB_UW3) {
            const int s = pos ? 1 : -1;
            if constexpr (RT)  // the taps nearly cancel: on differences the products stay small, and so do their roundings
              acc = vfma(tm, gk, vfma(tn, vsub(fk[-s], gk), vfma(tf, vsub(fk[-2 * s], gk), vmul(td, vsub(fk[s], gk)))));
            else
              acc = (tf * fk[-2 * s] + tn * fk[-s]) + (tm * gk + td * fk[s]);
          } else {  // WENO5 reconstructs the full J f; its rows of J come from the coefficient table
            const T fref = a.n0 * ac.ww[i][j];
            T x[7];
#pragma unroll
            for (int d = 0; d < 7; ++d)
              x[d] = a.coef[(int64_t)C_J * nt + axi_wrap(r0 + row + d - 3, nt)] * (fk[d - 3] + fref);
            const T D = pos ? weno_diff<T, true>(x) : weno_diff<T, false>(x);
            acc = -(vi * rv.ct) * D;
          }
          // force and inertial terms: (Gamma v_j^2 - F^theta) dg/dv_theta + sum_m K_jm h_m,
          // h_m = -Gamma v_i v_m g_im
          const T dvt = (K0 * g[j] + K1 * g[4 + j]) + (K2 * g[8 + j] + K3 * g[12 + j]);
          const T dvp = (ac.K[j][0] * (hb * fi[0]) + ac.K[j][1] * (ha * fi[P])) -
                        (ac.K[j][2] * (ha * fi[2 * P]) + ac.K[j][3] * (hb * fi[3 * P]));
          acc += (((j == 0 || j == 3) ? gb2 : ga2) - Ft) * dvt + dvp;
          const T xi = vfma(ac.v[j], up, ai);
          const T pm1 = vfma(xi, vfma(xi, vfma(xi, T(1.0 / 6.0), T(0.5)), c0), hu);
          acc = vadd(acc, vfma(-itau, gk, vmul(ac.ww[i][j], vfma(ntau, pm1, ci))));
          const T g0 = u0[(k0 + j) * P];
          o[j] = st == 0 ? gk + acc : g0 + b * ((gk - g0) + acc);
        }
        if (i == 0) {  // Cahn-Hilliard (Eq. CH): M Delta mu - div(u phi), theta parts only
          const T jp = RT ? rt[E_JP] : rv.jp, jm = RT ? rt[E_JM] : rv.jm;
          T L = (RT ? rt[E_LT] : rv.lt) * (jp * (mu_n - mu_c) - jm * (mu_c - mu_s));
          if (CH == VLB_HYDRO)
            L -= (RT ? rt[E_XN] : rv.xn) * (s_ut[m + 1] * ph[1]) - (RT ? rt[E_XS] : rv.xs) * (s_ut[m - 1] * ph[-1]);
          const T p0 = ph[0], lo = DF ? ph[P] : T(0);
          T bs = p0, bl = lo, inc = L;
          if (st > 0) {
            bs = u0[NPOP * P];
            bl = DF ? u0[(NPOP + 1) * P] : T(0);
            inc = b * (((p0 - bs) + (lo - bl)) + L);
          }
          if constexpr (DF) {  // (hi, lo) <- (base, base_lo) + inc, error-free sum, renormalised
            const T s1 = __fadd_rn(bs, inc), bb = __fsub_rn(s1, bs);
            const T lo2 = __fadd_rn(bl, __fadd_rn(__fsub_rn(bs, __fsub_rn(s1, bb)), __fsub_rn(inc, bb)));
            const T hi = __fadd_rn(s1, lo2);
            o[4] = hi;
            o[5] = __fsub_rn(lo2, __fsub_rn(hi, s1));
          } else {
            o[4] = bs + inc;
          }
          nout = DF ? 6 : 5;
        }
#pragma unroll
        for (int e = 0; e < 6; ++e) {
          if (e >= nout) break;
          const int k = e < 4 ? k0 + e : NPOP + e - 4;
          out[k * P + H + row] = o[e];
          const uint32_t off = (uint32_t)(ob * SZ + k * P + H + row);
          if (row < H) push(to_prev + (off + shift_prev) * (uint32_t)sizeof(T), o[e], bar_prev + 8u * par);
          if (row >= R - H) push(to_next + (off + shift_next) * (uint32_t)sizeof(T), o[e], bar_next + 8u * par);
        }
      }
      ok = mbar_wait1(bar + par, phase) && mbar_wait1(bar + 2 + par, phase);
      ok = __syncthreads_and(ok);
      if (!ok) break;
    }
  }
  if (!ok && tid == 0 && a.err) atomicExch(a.err, 2);  // a push never landed: flagged, the CTA winds down
  cluster_barrier();  // no CTA leaves while a neighbour may still push to it
  for (int k = 0; k < NST; ++k)
    for (int r = tid; r < R; r += kAxiThreads) U[k * a.stride + r0 + r] = buf[k * P + H + r];
}

// FP32 UW3 columns of at most kAxi16Rows rows per CTA: sixteen threads a row, one population each, which
// shortens the chain of a stage to about 0.7 us.  Same scheme of buffers, halos and pushes as axi_kernel; the
// groups of rows -1 and R only form moments and mu.  The row's constants and U^n stay in registers.  Above
// 30 rows a CTA the issue slots of one SM bind and four threads a row are as fast (32 rows: 6.2 against 4.6 us a
// step, both with cluster barriers); fewer CTAs are slower down to about eight rows each (64 rows on
// 1 / 4 / 8 CTAs: 4.6 / 2.9 / 2.5 us).
constexpr int kAxi16Rows = 30;

__host__ __device__ __forceinline__ size_t axi16_smem(int nt, int nc) {
  const int rmax = axi_count(nt, nc, 0);
  return sizeof(float) * (8 + (size_t)3 * (NARR + 1) * axi_pitch<float>(rmax, 2) + 2 * (size_t)(rmax + 2));
}

template <int CH>
__global__ void __launch_bounds__(512) axi16_kernel(StageArgs<float> a, const __grid_constant__ AxiConst<float> ac,
                                                     float* U, int steps) {
  constexpr int H = 2, NST = NARR + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nt = a.nt, nc = gridDim.x, c = blockIdx.x, tid = threadIdx.x;  // one cluster: rank = blockIdx.x
  const int r0 = axi_first(nt, nc, c), R = axi_count(nt, nc, c), rmax = axi_count(nt, nc, 0);
  const int P = axi_pitch<float>(rmax, H), SZ = NST * P;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);  // [from prev, from next][parity of the stage]
  float* buf = reinterpret_cast<float*>(smem_raw) + 8;
  float *s_mu = buf + 3 * SZ, *s_ut = s_mu + rmax + 2;
  for (int k = 0; k < NST; ++k)
    for (int r = tid; r < R + 2 * H; r += blockDim.x) buf[k * P + r] = U[k * a.stride + axi_wrap(r0 + r - H, nt)];
  const int cp = c > 0 ? c - 1 : nc - 1, cn = c + 1 < nc ? c + 1 : 0;
  const uint32_t base = smem_addr(buf);
  const int grp = min(tid >> 4, R + 1), k = tid & 15, i = k >> 2, j = k & 3;  // surplus groups repeat row R
  const bool own = grp >= 1 && grp <= R && (tid >> 4) <= R;
  const bool to_p = own && grp - 1 < H, to_n = own && grp - 1 >= R - H;
  const uint32_t prev = remote_addr(base, cp) + 4u * (uint32_t)(axi_count(nt, nc, cp)), next = remote_addr(base, cn) - 4u * (uint32_t)R;
  const bool pos = i >= 2;
  const float vi = ac.v[i], vj = ac.v[j], av = pos ? vi : -vi, ww = ac.ww[i][j], itau = a.inv_tau * a.dt;
  const float* rt = a.rows + (int64_t)axi_wrap(r0 + grp - 1, nt) * kRowTable;
  const bool bi = i == 0 || i == 3, bj = j == 0 || j == 3;
  const float* t = rt + E_TH + (bi ? 0 : 8);
  const float tf = t[pos ? TAP_FARP : TAP_FARN], tn = t[pos ? TAP_NEARP : TAP_NEARN];
  const float td = t[pos ? TAP_DOWNP : TAP_DOWNN];
  // the sum of the four taps, v_i (E + Gamma)
  const float gv = bi ? rt[E_GBB] / ac.v[3] : rt[E_GAA] / ac.v[2];
  const float ts = __fadd_rn(__fmaf_rn(vi, rt[E_EM], bi ? rt[E_NEB] : rt[E_NEA]), pos ? gv : -gv);
  const float gvj = bj ? rt[E_GBB] : rt[E_GAA], nv = a.n0 * vi, ce = a.n0 * (vi * rt[E_EM] + (bi ? rt[E_NEB] : rt[E_NEA]));
  const float lt = rt[E_LT], xn = rt[E_XN], xs = rt[E_XS], kt = rt[E_KT], jp = rt[E_JP], jm = rt[E_JM];
  const float avj = bj ? ac.v[3] : ac.v[2];
  float Kt[4], Kp[4];  // K_im, and -Gamma v_i v_m K_jm
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const float gvv = bi ? (m == 0 || m == 3 ? rt[E_GBB] : rt[E_GBA]) : (m == 0 || m == 3 ? rt[E_GBA] : rt[E_GAA]);
    Kt[m] = ac.K[i][m];
    Kp[m] = ac.K[j][m] * ((m >= 2) == pos ? -gvv : gvv);
  }
  const int sgn = pos ? 1 : -1;
  const float gt = a.gt * a.dt;
  const int at = k * P + H + grp - 1, ph_at = NPOP * P + H + grp - 1;
  // pushes to a neighbour complete on its barrier for data from this side
  const uint32_t bar_prev = remote_addr(smem_addr(bar + 2), cp), bar_next = remote_addr(smem_addr(bar), cn);
  float u0 = 0.0f, u0p = 0.0f, u0l = 0.0f;
  if (tid == 0) {
    for (int x = 0; x < 4; ++x) mbar_init1(bar + x);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  cluster_barrier();
  uint32_t stage = 0;
  bool ok = true;
  for (int n = 0; n < steps && ok; ++n) {
#pragma unroll
    for (int st = 0; st < 3; ++st, ++stage) {
      const uint32_t par = stage & 1;
      if (tid == 0) {  // armed before this CTA's own pushes, which let the neighbours run one stage ahead
        mbar_expect(bar + par, H * NST * 4);
        mbar_expect(bar + 2 + par, H * NST * 4);
      }
      const float* in = buf + st * SZ;
      const int ob = (st == 2 ? 0 : st + 1) * SZ;
      const float b = st == 1 ? 0.25f : 2.0f / 3.0f;
      const float g = in[at];
      const float* ph = in + ph_at;
      const float p0 = ph[0], lo = ph[P], pn = ph[1], ps = ph[-1];
      const float dN = (pn - p0) + (ph[P + 1] - lo), dS = (p0 - ps) + (lo - ph[P - 1]);
      // sums over j, then over i, each in the opposite pairs first (v_1 = -v_4, v_2 = -v_3)
      const float gx = __shfl_xor_sync(0xffffffffu, g, 3);
      float dn = g + gx, mp = avj * (j >= 2 ? g - gx : gx - g);
      dn += __shfl_xor_sync(0xffffffffu, dn, 1);
      mp += __shfl_xor_sync(0xffffffffu, mp, 1);
      const float dx = __shfl_xor_sync(0xffffffffu, dn, 12);
      float mt = av * (pos ? dn - dx : dx - dn);
      dn += dx;
      mp += __shfl_xor_sync(0xffffffffu, mp, 12);
      dn += __shfl_xor_sync(0xffffffffu, dn, 4);
      mt += __shfl_xor_sync(0xffffffffu, mt, 4);
      mp += __shfl_xor_sync(0xffffffffu, mp, 4);
      const float nn = __fadd_rn(a.n0, dn), inv_n = __frcp_rn(nn);
      const float ut = node_velocity(mt, inv_n, ac.fix), up = node_velocity(mp, inv_n, ac.fix);
      const float cubic = p0 * (1.0f - p0 * p0) + (1.0f - 3.0f * p0 * p0) * lo;  // at hi + lo, first order in lo
      const float mu_c = -a.A * cubic - kt * (jp * dN - jm * dS);
      if (k == 0) {
        s_mu[grp] = mu_c;
        s_ut[grp] = ut;
      }
      if (st == 0) {
        u0 = g;
        u0p = p0;
        u0l = lo;
      }
      __syncthreads();
      if (own) {
        const float mu_n = s_mu[grp + 1], mu_s = s_mu[grp - 1];
        float Ft = 0.0f;
        if (CH == VLB_HYDRO) Ft = p0 * inv_n * (mu_s - mu_n) * gt;  // n F^theta = -phi d_theta mu (Eq. pbin)
        const float* fk = in + at;
        const float* fr = in + H + grp - 1;
        // the taps nearly cancel: on differences the products stay small, and so do their roundings
        float acc = __fmaf_rn(tn, __fsub_rn(fk[-sgn], g), __fmul_rn(tf, __fsub_rn(fk[-2 * sgn], g)));
        float ac2 = __fmaf_rn(ts, g, __fmul_rn(td, __fsub_rn(fk[sgn], g)));
        // force and inertial terms: (Gamma v_j^2 - F^theta) dg/dv_theta - Gamma v_i sum_m K_jm v_m g_im
        const float dvt = (Kt[0] * fr[j * P] + Kt[1] * fr[(4 + j) * P]) + (Kt[2] * fr[(8 + j) * P] + Kt[3] * fr[(12 + j) * P]);
        const float* fi = fr + 4 * i * P;
        acc += Kp[0] * fi[0] + Kp[1] * fi[P];
        ac2 += Kp[2] * fi[2 * P] + Kp[3] * fi[3 * P];
        // n / tau from the density that was inverted for u: n0 / tau rounded on its own would be off by the same amount
        // at every node and stage, and the momentum would drift by it.  F^theta, the last to arrive, enters late.
        const float usq = ut * ut + up * up, hu = -0.5f * usq, xi = __fmaf_rn(vj, up, __fmul_rn(vi, ut));
        const float dntau = __fmul_rn(dn, itau), ntau = __fmul_rn(nn, itau);
        const float pm1 = __fmaf_rn(xi, __fmaf_rn(xi, __fmaf_rn(xi, 1.0f / 6.0f, 0.5f), 1.0f + hu), hu);
        const float X = __fmaf_rn(nv, Ft, __fmaf_rn(ntau, pm1, __fadd_rn(dntau, ce)));
        acc = __fmaf_rn(-Ft, dvt, __fmaf_rn(gvj, dvt, acc));
        acc = __fadd_rn(acc, __fmaf_rn(ww, X, __fmaf_rn(-itau, g, ac2)));
        const float o = st == 0 ? g + acc : u0 + b * ((g - u0) + acc);
        // Cahn-Hilliard (Eq. CH): M Delta mu - div(u phi), theta parts only (every lane; 0 and 1 store hi, lo)
        float L = lt * (jp * (mu_n - mu_c) - jm * (mu_c - mu_s));
        if (CH == VLB_HYDRO) L -= xn * (s_ut[grp + 1] * pn) - xs * (s_ut[grp - 1] * ps);
        const float bs = st == 0 ? p0 : u0p, bl = st == 0 ? lo : u0l;
        const float inc = st == 0 ? L : b * (((p0 - bs) + (lo - bl)) + L);
        const float s1 = __fadd_rn(bs, inc), bb = __fsub_rn(s1, bs);  // (hi, lo) <- (base, base_lo) + inc, error-free
        const float lo2 = __fadd_rn(bl, __fadd_rn(__fsub_rn(bs, __fsub_rn(s1, bb)), __fsub_rn(inc, bb)));
        const float hi = __fadd_rn(s1, lo2), pv = k == 0 ? hi : __fsub_rn(lo2, __fsub_rn(hi, s1));
        buf[ob + at] = o;
        if (k < 2) buf[ob + ph_at + k * P] = pv;
        if (to_p) {
          push(prev + 4u * (uint32_t)(ob + at), o, bar_prev + 8u * par);
          if (k < 2) push(prev + 4u * (uint32_t)(ob + ph_at + k * P), pv, bar_prev + 8u * par);
        }
        if (to_n) {
          push(next + 4u * (uint32_t)(ob + at), o, bar_next + 8u * par);
          if (k < 2) push(next + 4u * (uint32_t)(ob + ph_at + k * P), pv, bar_next + 8u * par);
        }
      }
      const uint32_t phase = (stage >> 1) & 1;
      ok = mbar_wait1(bar + par, phase) && mbar_wait1(bar + 2 + par, phase);
      ok = __syncthreads_and(ok);
      if (!ok) break;
    }
  }
  if (!ok && tid == 0 && a.err) atomicExch(a.err, 2);  // a push never landed: flagged, the CTA winds down
  cluster_barrier();  // no CTA leaves while a neighbour may still push to it
  for (int q = 0; q < NST; ++q)
    for (int r = tid; r < R; r += blockDim.x) U[q * a.stride + r0 + r] = buf[q * P + H + r];
}

template <typename T>
AxiConst<T> make_axi_const() {
  const VelocityConsts d = velocity_consts();
  AxiConst<T> c;
  for (int i = 0; i < 4; ++i) {
    c.v[i] = (T)d.v[i];
    for (int m = 0; m < 4; ++m) {
      c.K[i][m] = (T)d.K[i][m];
      c.ww[i][m] = (T)(d.w[i] * d.w[m]);
    }
  }
  c.fix = make_node_const<T>().fix;
  return c;
}

cudaLaunchConfig_t axi_config(int nc, int threads, size_t smem, cudaStream_t st, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nc);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = nc;
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// CTAs a cluster of this kernel may have on the current device (once per kernel and device: the opt-in to
// shared memory and, if the device takes it, to the non-portable cluster size)
template <typename K>
cudaError_t axi_most(K kernel, int (&most)[32], int* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 32) return cudaErrorInvalidDevice;
  if (most[dev] == 0) {
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax)) != cudaSuccess)
      return e;
    int m = kAxiPortable, n = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
      cudaLaunchAttribute attr[1];
      const cudaLaunchConfig_t cfg = axi_config(kAxiCta, kAxiThreads, kSmemMax, nullptr, attr);
      if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n >= 1) m = kAxiCta;
    }
    cudaGetLastError();  // a refused opt-in leaves the portable size
    most[dev] = m;
  }
  *out = most[dev];
  return cudaSuccess;
}

template <typename T, int ADV, int CH>
cudaError_t launch_axi_t(const StageArgs<T>& a, T* U, int steps, cudaStream_t st) {
  static const AxiConst<T> ac = make_axi_const<T>();
  cudaLaunchAttribute attr[1];
  cudaError_t e;
  int nc = 0;
  if constexpr (sizeof(T) == 4 && ADV == VLB_UW3) {
    static int most16[32] = {0};
    if ((e = axi_most(axi16_kernel<CH>, most16, &nc)) != cudaSuccess) return e;
    if (a.route & VLB_TEST_PORTABLE_CLUSTER) nc = kAxiPortable;
    nc = std::min(nc, std::max(1, a.nt / 8));
    const int rows = axi_count(a.nt, nc, 0);
    if (rows <= kAxi16Rows) {
      const cudaLaunchConfig_t cfg = axi_config(nc, ((rows + 2) * 16 + 31) / 32 * 32, axi16_smem(a.nt, nc), st, attr);
      return cudaLaunchKernelEx(&cfg, axi16_kernel<CH>, a, ac, U, steps);
    }
  }
  static int most[32] = {0};
  if ((e = axi_most(axi_kernel<T, ADV, CH>, most, &nc)) != cudaSuccess) return e;
  if (a.route & VLB_TEST_PORTABLE_CLUSTER) nc = kAxiPortable;
  nc = std::min(nc, std::max(1, a.nt / 4));
  const bool table = axi_smem<T, ADV>(a.nt, nc, true) <= kSmemMax;
  const size_t smem = axi_smem<T, ADV>(a.nt, nc, table);
  if (smem > kSmemMax) return cudaErrorInvalidValue;  // never: see the assertion at axi_smem
  const cudaLaunchConfig_t cfg = axi_config(nc, kAxiThreads, smem, st, attr);
  return cudaLaunchKernelEx(&cfg, axi_kernel<T, ADV, CH>, a, ac, U, steps, table ? 1 : 0);
}

}  // namespace

template <typename T>
cudaError_t launch_axi(const StageArgs<T>& a, int advection, int ch_mode, T* U, int steps, cudaStream_t s) {
  if (a.ns != 1 || a.nt < 4 || a.nt > kAxiMaxRows || steps < 0) return cudaErrorInvalidValue;
  if (steps == 0) return cudaSuccess;
  if (advection == VLB_UW3)
    return ch_mode == VLB_HYDRO ? launch_axi_t<T, VLB_UW3, VLB_HYDRO>(a, U, steps, s)
                                : launch_axi_t<T, VLB_UW3, VLB_DIFFUSIVE>(a, U, steps, s);
  return ch_mode == VLB_HYDRO ? launch_axi_t<T, VLB_WENO5, VLB_HYDRO>(a, U, steps, s)
                              : launch_axi_t<T, VLB_WENO5, VLB_DIFFUSIVE>(a, U, steps, s);
}

template cudaError_t launch_axi<float>(const StageArgs<float>&, int, int, float*, int, cudaStream_t);
template cudaError_t launch_axi<double>(const StageArgs<double>&, int, int, double*, int, cudaStream_t);

}  // namespace vlb
