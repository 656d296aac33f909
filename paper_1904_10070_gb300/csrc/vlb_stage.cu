// Fused Runge-Kutta stage of the vielbein LB + Cahn-Hilliard solver (arXiv:1904.10070).
//
// One launch evaluates, for every node of the periodic (theta, varphi) grid,
//   L_f   = right-hand side of Eq. boltz_tor with BGK collisions (Sec. 2.3),
//   L_phi = right-hand side of Eq. CH with mu from Eq. mu and the force of Eq. pbin,
// and writes U_out = U^n + b (U_in - U^n + dt L(U_in)) -- one stage of SSP-RK3 in Shu-Osher form
// (b = 1, 1/4, 2/3), written so that the weights only multiply small increments.  The populations
// are stored as deviations g = f - n0 w_i w_j from the rest equilibrium, and in FP32 mode phi is
// carried as an unevaluated float pair hi + lo (vlb_internal.cuh explains both).
//
// Work unit: a tile of TQ theta rows x 32 varphi columns.  For a tile the CTA
//   1. stages, with asynchronous global->shared copies (cp.async), a box of H = 2 rows
//      and HS columns around the tile for the 16 populations and phi, the tile's
//      U^n values and the per-row coefficients;
//   2. computes the moments and mu on the tile plus a halo of 1;
//   3. computes the right-hand sides and the Runge-Kutta combination and stores the tile.
// One 128-thread CTA per 8 x 32 tile, four CTAs per SM, or one 256-thread CTA per 16 x 32 tile, two per SM
// (stage_rows_rule).  For FP32 UW3 grids with n_phi % 4 == 0 (the
// production path) steps 2 and 3 run on adjacent node pairs in packed FP32x2 arithmetic, two lanes of
// one float2 per thread: a thread loads its pair once in step 2, keeps the parity combinations of the
// populations (vlb_node.cuh) over the barrier and reads everything that depends on the row from a table.
// The stage is bound by latency and the shared-memory pipe at 16 warps per SM (issue slots 45% busy), with HBM at
// about 80%.  A stage at 1024 x 2048, first / later ones: 77.7 / 82.6 us on the populations themselves, 68.6 / 76.1
// in the parity basis (44.0 against 34.0 M warp instructions), 62.8 / 73.5 with 8-row tiles, which fit four to an SM
// because step 3 sums dn again and phi of U^n comes from L2; per step 0.235, 0.217 and 0.204 ms.
// Ragged ensemble members run steps 2 and 3 in scalar arithmetic, two nodes per thread.  A persistent double-
// buffered variant (next tile copied in while the current one computes, one 384-thread CTA per SM) measured 1.6x
// slower on GB300: with
// 12 warps per SM and all warps issuing copies and shared loads in the same phase, the memory-
// input queue throttled issue to 30%.  FP64 and WENO5 grids and FP32 UW3 grids off the packed layout are stepped
// by direct_kernel (vlb_direct.cu).
// Periodic wrap-around is resolved on the copy addresses, so ragged tiles need no special case.
#include <vector>

#include "vlb_node.cuh"

namespace vlb {

namespace {

constexpr int TS = 32;   // tile width along varphi
constexpr int NCT = 11;  // coefficient rows staged in shared memory (C_J .. C_EN)

struct VConst {
  float v[4], w[4], K[4][4];
  float ww[4][4];  // w_i w_j
  NodeConst<float> nc;
};

// Shared-memory layout of one CTA of TQ rows.  Offsets are in floats.
template <int TQ_>
struct StageLayR {
  static constexpr int H = 2, TQ = TQ_, HS = 4, NTH = TQ * (TS / 2);  // halo rows, halo columns staged, threads
  static constexpr int NST = NARR + 1;  // state arrays (= staged boxes): populations, phi, phi lo
  // arrays of the staged U^n tile: with 16 rows phi too (two CTAs per SM either way; from L2 it is a wait of its own in
  // every tile, 0.50 against 0.45 ms a step in the wavefront schedule), with 8 rows from L2, to fit four CTAs
  static constexpr int NU0 = TQ == 16 ? NST : NPOP;
  static constexpr int BQ = TQ + 2 * H, BS = TS + 2 * HS;
  static constexpr int BOX = NST * BQ * BS;
  // moment / mu box: halo 1, column origin -2; column TS of a row takes the next row's unused column -2
  static constexpr int MQ = TQ + 2, MS = TS + 2, MN = MQ * MS + 2;
  // row coefficients: NCT x BQ for the scalar step 3, or the row table of rows -1 .. TQ for packed pairs; padded:
  // sub-buffers stay 128-byte aligned
  static constexpr int CO = ((NCT * BQ > (TQ + 2) * kRowTable ? NCT * BQ : (TQ + 2) * kRowTable) + 31) / 32 * 32;
  static constexpr int VEC = 4;  // floats per 16-byte chunk
  static constexpr int CO_OFF = BOX;
  static constexpr int U0_OFF = CO_OFF + CO;
  static constexpr int UT_OFF = U0_OFF + NU0 * TQ * TS;
  static constexpr int UP_OFF = UT_OFF + MN;
  static constexpr int MU_OFF = UP_OFF + MN;
  static constexpr int MB_OFF = (MU_OFF + MN + 1) / 2 * 2;  // two 8-byte mbarriers
  static constexpr int TOTAL = MB_OFF + 4;
  static constexpr size_t BYTES = sizeof(float) * (size_t)TOTAL;
  static_assert(BOX % VEC == 0 && BS % VEC == 0 && HS % VEC == 0 && CO_OFF % VEC == 0 && U0_OFF % VEC == 0,
                "box rows, tile columns and sub-buffers start on a 16-byte boundary");
};
using StageLay = StageLayR<16>;

__device__ __forceinline__ int wrap(int x, int n) {
  x %= n;
  return x < 0 ? x + n : x;
}

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst)), "l"(src));
}

__device__ __forceinline__ void cp_async_small(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_u32(dst)), "l"(src));
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }

template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Programmatic dependent launch: a stage may start while the previous kernel in the stream drains.
// pdl_wait() blocks until that kernel has completed and its writes are visible (a no-op without a
// programmatic launch); pdl_trigger() lets the next stage's CTAs be scheduled.  Every global
// access (state buffers and coefficient tables) comes after pdl_wait(); only shared-memory set-up
// runs before it.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

// mbarrier and bulk tensor copy (TMA) primitives.
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: gives up after 2^22 polls (each poll may suspend the thread for a while), so that a
// copy that never lands cannot hang the GPU.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity) {
  for (int it = 0; it < (1 << 22); ++it)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}
// Copy the box {x, y, z} .. + box dims of a 3-D tensor map into shared memory (128-byte aligned),
// completing on bar.
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], "
      "[%2];\n" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
      : "memory");
}

// Prefetch the box {x, y, z} .. + box dims of a 3-D tensor map into L2 (a hint: no shared memory).
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap* map, int x, int y, int z) {
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];\n" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y), "r"(z)
               : "memory");
}

__device__ __forceinline__ float recip(float x) { return __frcp_rn(x); }

// Whether the chunked copy path applies: rows wrap at most once and columns come in aligned
// 16-byte chunks that never straddle the periodic seam.
template <typename L>
__host__ __device__ inline bool chunked(int nt, int ns) {
  return ns % L::VEC == 0 && ns >= L::BS && nt >= L::BQ;
}

// ---------------------------------------------------------------------------------------------
// Step 1: asynchronous copies of the box (populations and phi of U_in) with its row coefficients,
// and of the tile's U^n.
// ---------------------------------------------------------------------------------------------
template <typename L>
__device__ __forceinline__ void issue_co(const StageArgs<float>& a, float* co, int q0, int tid) {
  for (int idx = tid; idx < NCT * L::BQ; idx += L::NTH) {
    const int k = idx / L::BQ, r = idx - k * L::BQ;
    cp_async_small(co + idx, a.coef + (int64_t)k * a.nt + wrap(q0 + r - L::H, a.nt));
  }
}

template <typename L>
__device__ __forceinline__ void issue_box(const StageArgs<float>& a, float* box, float* co, int q0, int s0, int tid) {
  constexpr int H = L::H, BQ = L::BQ, BS = L::BS, HS = L::HS;
  constexpr int VEC = L::VEC;
  const int nt = a.nt, ns = a.ns;
  const int64_t stride = a.stride;
  if (chunked<L>(nt, ns)) {
    constexpr int CPR = BS / VEC;  // 16-byte chunks of a box row
    for (int pos = tid; pos < BQ * CPR; pos += L::NTH) {
      const int r = pos / CPR, col = (pos - r * CPR) * VEC;
      int gq = q0 + r - H;
      gq += gq < 0 ? nt : (gq >= nt ? -nt : 0);
      int gs = s0 - HS + col;
      gs += gs < 0 ? ns : (gs >= ns ? -ns : 0);
      const float* src = a.fin + (int64_t)gq * ns + gs;
      float* dst = box + r * BS + col;
#pragma unroll
      for (int k = 0; k < L::NST; ++k) cp_async16(dst + k * BQ * BS, src + k * stride);
    }
  } else {
    for (int idx = tid; idx < L::NST * BQ * BS; idx += L::NTH) {
      const int k = idx / (BQ * BS);
      const int rem = idx - k * (BQ * BS);
      const int r = rem / BS, c = rem - r * BS;
      const int gq = wrap(q0 + r - H, nt), gs = wrap(s0 + c - HS, ns);
      cp_async_small(box + (k * BQ + r) * BS + c, a.fin + k * stride + (int64_t)gq * ns + gs);
    }
  }
}

template <typename L>
__device__ __forceinline__ void issue_u0(const StageArgs<float>& a, float* su0, int q0, int s0, int tid) {
  constexpr int TQ = L::TQ, VEC = L::VEC;
  const int nt = a.nt, ns = a.ns;
  const int64_t stride = a.stride;
  if (chunked<L>(nt, ns)) {
    // TQ x TS/VEC chunk positions; the arrays are split between groups of threads
    constexpr int CT = TS / VEC, NPOS = TQ * CT;
    constexpr int GROUPS = L::NTH / NPOS > 0 ? L::NTH / NPOS : 1;
    constexpr int PER = (L::NU0 + GROUPS - 1) / GROUPS;
    for (int t = tid; t < NPOS * GROUPS; t += L::NTH) {
      const int pos = t % NPOS, grp = t / NPOS;
      const int r = pos / CT, ch = pos - r * CT;
      const int gq = q0 + r, gs = s0 + ch * VEC;
      if (gq < nt && gs < ns) {
        const float* src = a.f0 + (int64_t)gq * ns + gs;
        float* dst = su0 + r * TS + ch * VEC;
        const int k0 = grp * PER, k1 = k0 + PER < L::NU0 ? k0 + PER : L::NU0;
#pragma unroll 4
        for (int k = k0; k < k1; ++k) cp_async16(dst + k * TQ * TS, src + k * stride);
      }
    }
  } else {
    for (int idx = tid; idx < L::NU0 * TQ * TS; idx += L::NTH) {
      const int k = idx / (TQ * TS);
      const int rem = idx - k * (TQ * TS);
      const int r = rem / TS, c = rem - r * TS;
      const int gq = q0 + r, gs = s0 + c;
      if (gq < nt && gs < ns)
        cp_async_small(su0 + (k * TQ + r) * TS + c, a.f0 + k * stride + (int64_t)gq * ns + gs);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Step 2: moments (Sec. 2.3) and mu (Eq. mu) on the tile plus a halo of 1 (cross-shaped).
// Moment-box position (mr, mc) is tile node (mr - 1, mc - 2).
// ---------------------------------------------------------------------------------------------
// Moments and mu at moment-box position (mr, mc).
template <typename L>
__device__ __forceinline__ void moment_point(const StageArgs<float>& a, const VConst& vc, const float* box, const float* co,
                                             float* sm, int mr, int mc) {
  constexpr int H = L::H, BQ = L::BQ, BS = L::BS, HS = L::HS, MS = L::MS;
  const float* sf = box;
  const float* sphi = box + NPOP * BQ * BS;
  const float* sphl = box + (NPOP + 1) * BQ * BS;
  const int bi = (mr + H - 1) * BS + (mc - 2 + HS);  // box index of this position
  const float* fp = sf + bi;
  float row[4] = {0.0f, 0.0f, 0.0f, 0.0f}, col[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float x = fp[(4 * i + j) * BQ * BS];
      row[i] += x;
      col[j] += x;
    }
  // n = n0 + sum g (the reference part carries no momentum); v_1 = -v_4, v_2 = -v_3
  const float dn = (row[0] + row[1]) + (row[2] + row[3]);
  const float mt = vc.v[3] * (row[3] - row[0]) + vc.v[2] * (row[2] - row[1]);
  const float mp = vc.v[3] * (col[3] - col[0]) + vc.v[2] * (col[2] - col[1]);
  const int mi = mr * MS + mc;
  const float inv_n = recip(a.n0 + dn);
  sm[L::UT_OFF + mi] = node_velocity(mt, inv_n, vc.nc.fix);
  sm[L::UP_OFF + mi] = node_velocity(mp, inv_n, vc.nc.fix);
  const float* pp = sphi + bi;
  const int cr = mr + H - 1;
  const float ph = pp[0];
  // neighbour differences of phi = hi + lo: the hi differences are exact for nearby values
  float dN = pp[BS] - ph, dS = ph - pp[-BS], dE = pp[1] - ph, dW = ph - pp[-1];
  const float* pl = sphl + bi;
  const float lo = pl[0];
  dN += pl[BS] - lo;
  dS += lo - pl[-BS];
  dE += pl[1] - lo;
  dW += lo - pl[-1];
  const float lap = co[C_LT * BQ + cr] * (co[C_JP * BQ + cr] * dN - co[C_JM * BQ + cr] * dS) +
                    co[C_LP * BQ + cr] * (dE - dW);
  // phi (1 - phi^2) at hi + lo, to first order in lo
  const float cubic = ph * (1.0f - ph * ph) + (1.0f - 3.0f * ph * ph) * lo;
  sm[L::MU_OFF + mi] = -a.A * cubic - a.kappa * lap;
}

template <typename L>
__device__ __forceinline__ void phase2(const StageArgs<float>& a, const VConst& vc, const float* box, const float* co,
                                       float* sm, int tid) {
  constexpr int MQ = L::MQ, TQ = L::TQ;
  constexpr int MS2 = TS + 2;  // tile columns -1 .. TS in the rows of the tile
  constexpr int PA = TQ * MS2;
  constexpr int PM = PA + 2 * TS;
  for (int idx = tid; idx < PM; idx += L::NTH) {
    int mr, mc;
    if (idx < PA) {
      mr = 1 + idx / MS2;
      mc = 1 + (idx - (mr - 1) * MS2);
    } else {
      const int j = idx - PA;
      mr = (j < TS) ? 0 : MQ - 1;
      mc = 2 + (j < TS ? j : j - TS);
    }
    moment_point<L>(a, vc, box, co, sm, mr, mc);
  }
}

// ---------------------------------------------------------------------------------------------
// Step 3, scalar: right-hand sides and the Runge-Kutta combination for node (lr, lc) of the tile.
// ---------------------------------------------------------------------------------------------
template <typename L, int CH, bool F0>
__device__ __forceinline__ void phase3_node(const StageArgs<float>& a, const VConst& vc, const float* box, const float* co,
                                            const float* sm, int lr, int lc, int q, int s) {
  constexpr int H = L::H, BQ = L::BQ, BS = L::BS, HS = L::HS, MS = L::MS, TQ = L::TQ;
  const float* sf = box;
  const float* sphi = box + NPOP * BQ * BS;
  const float* sphl = box + (NPOP + 1) * BQ * BS;
  const float* su0 = sm + L::U0_OFF;
  const float* sut = sm + L::UT_OFF;
  const float* sup = sm + L::UP_OFF;
  const float* smu = sm + L::MU_OFF;
  const int64_t stride = a.stride;
  const float sixth = 1.0f / 6.0f;
  const int fr = lr + H, fc = lc + HS;
  const int bi = fr * BS + fc;
  const int mi = (lr + 1) * MS + (lc + 2);
  const int ui = lr * TS + lc;

  // population deviations at the node, and their sum as in step 2
  float g[NPOP], row[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int k = 0; k < NPOP; ++k) {
    g[k] = sf[k * BQ * BS + bi];
    row[k >> 2] += g[k];
  }
  const float dn = (row[0] + row[1]) + (row[2] + row[3]), ut = sut[mi], up = sup[mi], ph = sphi[bi];
  const float n = a.n0 + dn;
  const float ct = co[C_CT * BQ + fr], cp = co[C_CP * BQ + fr], gam = co[C_GAM * BQ + fr];
  const float mu_c = smu[mi], mu_n = smu[mi + MS], mu_s = smu[mi - MS], mu_e = smu[mi + 1], mu_w = smu[mi - 1];

  // Cahn-Hilliard: M Delta mu - div(u phi) (Eq. CH), flux form with mean face values
  float Lphi = a.M * (co[C_LT * BQ + fr] * (co[C_JP * BQ + fr] * (mu_n - mu_c) - co[C_JM * BQ + fr] * (mu_c - mu_s)) +
                  co[C_LP * BQ + fr] * (mu_e - 2.0f * mu_c + mu_w));
  float Ft = 0.0f, Fp = 0.0f;
  if (CH == VLB_HYDRO) {
    const float Xn = co[C_J * BQ + fr + 1] * sut[mi + MS] * sphi[bi + BS];
    const float Xs = co[C_J * BQ + fr - 1] * sut[mi - MS] * sphi[bi - BS];
    const float Ye = sup[mi + 1] * sphi[bi + 1];
    const float Yw = sup[mi - 1] * sphi[bi - 1];
    Lphi -= 0.5f * (ct * (Xn - Xs) + cp * (Ye - Yw));
    // n F = -phi grad mu (Eq. pbin), central differences
    const float pn = ph * recip(n);
    Ft = -pn * (mu_n - mu_s) * a.gt;
    Fp = -pn * (mu_e - mu_w) * co[C_GP * BQ + fr];
  }

  const int64_t gidx = (int64_t)q * a.ns + s;
  if (a.dphi) {
    a.dphi[gidx] = Lphi * a.dt;  // the stabilised Cahn-Hilliard solve forms phi
  } else {
    const float lo = sphl[bi];
    float base = ph, base_lo = lo, inc = Lphi * a.dt;
    if (F0) {
      base = L::NU0 > NPOP ? su0[NPOP * TQ * TS + ui] : __ldcg(a.f0 + NPOP * stride + gidx);
      base_lo = L::NU0 > NPOP ? su0[(NPOP + 1) * TQ * TS + ui] : __ldcg(a.f0 + (NPOP + 1) * stride + gidx);
      inc = a.b * (((ph - base) + (lo - base_lo)) + inc);
    }
    // (hi, lo) <- (base, base_lo) + inc with an error-free sum, then renormalised
    const float s1 = base + inc;
    const float bb = s1 - base;
    const float err = (base - (s1 - bb)) + (inc - bb);
    const float lo2 = base_lo + err;
    const float hi_out = s1 + lo2;
    a.fout[NPOP * stride + gidx] = hi_out;
    a.fout[(NPOP + 1) * stride + gidx] = lo2 - (hi_out - s1);
  }

  // UW3 advection weights: the theta flux difference of G = J g with ct/6 folded in, over
  // d = -2..1 (v > 0) and d = -1..2 (v < 0); the varphi difference is scaled by cp/6.
  const float ct6 = ct * sixth, cp6 = cp * sixth;
  const float Jm1 = co[C_J * BQ + fr - 1], J0 = co[C_J * BQ + fr], Jp1 = co[C_J * BQ + fr + 1];
  const float wp0 = ct6 * co[C_J * BQ + fr - 2], wp1 = -6.0f * ct6 * Jm1, wp2 = 3.0f * ct6 * J0, wp3 = 2.0f * ct6 * Jp1;
  const float wn0 = -2.0f * ct6 * Jm1, wn1 = -3.0f * ct6 * J0, wn2 = 6.0f * ct6 * Jp1, wn3 = -ct6 * co[C_J * BQ + fr + 2];

  const float usq = ut * ut + up * up;
  const float c0 = 1.0f - 0.5f * usq;
  const float hu = -0.5f * usq;
  const float ntau = n * a.inv_tau, dntau = dn * a.inv_tau;
  const float Ep = co[C_EP * BQ + fr], En = co[C_EN * BQ + fr];

#pragma unroll
  for (int i = 0; i < 4; ++i) {
    // varphi-derivative operands h_m = (-F^phi - Gamma v_i v_m) g_{i m}; K~ = K diag(v) (Sec. 2.3)
    const float gvi = gam * vc.v[i];
    float h[4];
#pragma unroll
    for (int mm = 0; mm < 4; ++mm) h[mm] = (-Fp - gvi * vc.v[mm]) * g[4 * i + mm];
    const float ai = vc.v[i] * ut;
    // The BGK relaxation and the closed-form reference part share the factor w_i w_j:
    //   (f^eq - n0 w w)/tau + n0 w w [v_i (E(q) + F^theta) + v_j F^phi]
    //   = w_i w_j [ (dn + n (poly - 1))/tau + n0 v_i (E + F^theta) + n0 v_j F^phi ]
    const float ci = dntau + a.n0 * vc.v[i] * ((i >= 2 ? Ep : En) + Ft);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = 4 * i + j;
      const float* fk = sf + k * BQ * BS + bi;
      const float Dt = (i >= 2) ? wp0 * fk[-2 * BS] + wp1 * fk[-BS] + wp2 * g[k] + wp3 * fk[BS]
                            : wn0 * fk[-BS] + wn1 * g[k] + wn2 * fk[BS] + wn3 * fk[2 * BS];
      const float Dp = (j >= 2) ? (fk[-2] - 6.0f * fk[-1] + 3.0f * g[k] + 2.0f * fk[1])
                            : (-2.0f * fk[-1] - 3.0f * g[k] + 6.0f * fk[1] - fk[2]);
      float rhs = -(vc.v[i] * Dt) - (vc.v[j] * cp6) * Dp;
      // force and inertial terms on the deviation: (Gamma v_j^2 - F^theta) dg/dv_theta + sum_m K_jm h_m
      float dvt = 0.0f, dvp = 0.0f;
#pragma unroll
      for (int mm = 0; mm < 4; ++mm) {
        dvt += vc.K[i][mm] * g[4 * mm + j];
        dvp += vc.K[j][mm] * h[mm];
      }
      rhs += (gam * vc.v[j] * vc.v[j] - Ft) * dvt + dvp;
      // BGK towards the third-order Hermite equilibrium (Eq. feq) plus the reference part
      const float xi = ai + vc.v[j] * up;
      const float pm1 = xi * (c0 + xi * (0.5f + xi * sixth)) + hu;
      const float X = ntau * pm1 + (ci + a.n0 * vc.v[j] * Fp);
      rhs += vc.ww[i][j] * X - a.inv_tau * g[k];
      float o;
      if (F0) {
        const float g0 = su0[k * TQ * TS + ui];
        o = g0 + a.b * ((g[k] - g0) + rhs * a.dt);
      } else {
        o = rhs * a.dt + g[k];
      }
      a.fout[k * stride + gidx] = o;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Packed FP32 pairs: two horizontally adjacent nodes per thread, one float2 lane each.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float2 f2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ void st2(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }

// (hi, lo) <- (base, base_lo) + inc with an error-free sum, renormalised (one lane)
__device__ __forceinline__ void df_add(float base, float base_lo, float inc, float& hi, float& lo) {
  const float s1 = base + inc;
  const float bb = s1 - base;
  const float err = (base - (s1 - bb)) + (inc - bb);
  const float lo2 = base_lo + err;
  hi = s1 + lo2;
  lo = lo2 - (hi - s1);
}

// (0, r): the row table of row q0 + r - 1, r = 0 .. TQ + 1, by 16-byte copies
template <typename L>
__device__ __forceinline__ void issue_rows(const StageArgs<float>& a, float* co, int q0, int tid) {
  for (int x = tid; x < (L::TQ + 2) * (kRowTable / 4); x += L::NTH) {
    const int r = x / (kRowTable / 4), c = x % (kRowTable / 4);
    cp_async16(co + r * kRowTable + 4 * c, a.rows + (int64_t)wrap(q0 + r - 1, a.nt) * kRowTable + 4 * c);
  }
}

// Moments, mu and the parity combinations of a pair of adjacent nodes.
struct PairNode {
  float2 P[16], dn, inv, ut, up, ph, lo, mu;
};

static_assert(E_JP % 4 == 0 && E_KP == E_JP + 3 && E_TH % 8 == 0 && NROW32 == kRowTable, "16-byte groups of the row table");

// Step 2 on packed node pairs (FP32): moment-box positions (mr, mc) and (mr, mc + 1), mc even.
template <typename L>
__device__ __forceinline__ void pair_point(const StageArgs<float>& a, const NodeConst<float>& nc, const float* box,
                                           const float* rows, int mr, int mc, PairNode& o) {
  constexpr int H = L::H, BQ = L::BQ, BS = L::BS, HS = L::HS, MS = L::MS;
  static_assert(HS % 2 == 0 && BS % 2 == 0 && MS % 2 == 0 && L::UT_OFF % 2 == 0 && L::UP_OFF % 2 == 0 &&
                    L::MU_OFF % 2 == 0,
                "pair alignment");
  const int bi = (mr + H - 1) * BS + (mc - 2 + HS);  // even
  const float* fp = box + bi;
#pragma unroll
  for (int k = 0; k < 16; ++k) o.P[k] = ld2(fp + k * BQ * BS);
  const float* pp = box + NPOP * BQ * BS + bi;
  const float* pl = box + (NPOP + 1) * BQ * BS + bi;
  const float2 ph = ld2(pp), lo = ld2(pl);
  const float2 phW = ld2(pp - 2), phE = ld2(pp + 2), loW = ld2(pl - 2), loE = ld2(pl + 2);
  // neighbour differences of phi = hi + lo: the hi differences are exact for nearby values
  float2 dN = vsub(ld2(pp + BS), ph), dS = vsub(ph, ld2(pp - BS));
  float2 dE = vsub(make_float2(ph.y, phE.x), ph), dW = vsub(ph, make_float2(phW.y, ph.x));
  dN = vadd(dN, vsub(ld2(pl + BS), lo));
  dS = vadd(dS, vsub(lo, ld2(pl - BS)));
  dE = vadd(dE, vsub(make_float2(lo.y, loE.x), lo));
  dW = vadd(dW, vsub(lo, make_float2(loW.y, lo.x)));
  const float4 c = *reinterpret_cast<const float4*>(rows + mr * kRowTable + E_JP);  // JP, JM, KT, KP
  const float2 klap = vfma(f2(c.w), vsub(dE, dW), vmul(f2(c.z), vsub(vmul(f2(c.x), dN), vmul(f2(c.y), dS))));
  // phi (1 - phi^2) at hi + lo, to first order in lo
  const float2 ph2 = vmul(ph, ph);
  const float2 cubic = vfma(vfma(f2(-3.0f), ph2, f2(1.0f)), lo, vmul(ph, vsub(f2(1.0f), ph2)));
  o.mu = vsub(vmul(f2(-a.A), cubic), klap);
  to_parity16(o.P);
  float2 mt, mp;
  parity_moments(o.P, nc, o.dn, mt, mp);
  const float2 nn = vadd(f2(a.n0), o.dn);
  o.inv = make_float2(__frcp_rn(nn.x), __frcp_rn(nn.y));
  o.ut = node_velocity(mt, o.inv, nc.fix);
  o.up = node_velocity(mp, o.inv, nc.fix);
  o.ph = ph;
  o.lo = lo;
}

// Step 2 for the whole tile.  A thread's own pair of nodes stays in registers for step 3 (with its parity
// combinations); the threads of the first warps also take the halo: rows -1 and TQ (mu, u^theta), and the
// columns -1 and TS inside the aligned pairs (-2, -1) and (TS, TS + 1), keeping one lane (mu, u^phi), so
// that every column takes the same sequence of FP32 operations (an axisymmetric state stays bitwise
// axisymmetric).  The pairs' other lanes read box columns -4 .. TS + 3, inside the HS = 4 halo.
template <typename L>
__device__ __forceinline__ void phase2_pair(const StageArgs<float>& a, const NodeConst<float>& nc, const float* box,
                                            const float* rows, float* sm, int tid, PairNode& own) {
  constexpr int MQ = L::MQ, TQ = L::TQ, MS = L::MS, NROWS = TS;  // TS / 2 pairs in each of two halo rows
  static_assert(L::HS >= 4, "the halo pairs read two columns beyond the halo column");
  static_assert(L::NTH == TQ * (TS / 2) && NROWS + 2 * TQ <= L::NTH, "one node pair per thread, one halo item at most");
  if (tid < NROWS + 2 * TQ) {
    PairNode h;
    if (tid < NROWS) {
      const int mr = tid < TS / 2 ? 0 : MQ - 1, mc = 2 + 2 * (tid % (TS / 2));
      pair_point<L>(a, nc, box, rows, mr, mc, h);
      st2(sm + L::MU_OFF + mr * MS + mc, h.mu);
      st2(sm + L::UT_OFF + mr * MS + mc, h.ut);
    } else {
      const int j = tid - NROWS, mr = 1 + (j >> 1);
      const bool east = j & 1;
      const int mc = east ? TS + 2 : 0, mi = mr * MS + mc + (east ? 0 : 1);
      pair_point<L>(a, nc, box, rows, mr, mc, h);
      sm[L::MU_OFF + mi] = east ? h.mu.x : h.mu.y;
      sm[L::UP_OFF + mi] = east ? h.up.x : h.up.y;
    }
  }
  const int mr = 1 + tid / (TS / 2), mc = 2 + 2 * (tid % (TS / 2));
  pair_point<L>(a, nc, box, rows, mr, mc, own);
  st2(sm + L::MU_OFF + mr * MS + mc, own.mu);
  st2(sm + L::UT_OFF + mr * MS + mc, own.ut);
  st2(sm + L::UP_OFF + mr * MS + mc, own.up);
}

// phi of U^n at a thread's pair of nodes, loaded before step 2 so that it is in flight meanwhile; from L2, since
// a persistent launch may hold a line of an earlier step in L1.  Not where the staged tile has it.
template <typename L, bool F0>
__device__ __forceinline__ void load_u0_phi(const StageArgs<float>& a, int q, int s, float2& hi, float2& lo) {
  if (L::NU0 == NPOP && F0 && !a.dphi && q < a.nt && s < a.ns) {
    const float* p = a.f0 + NPOP * a.stride + (int64_t)q * a.ns + s;
    hi = __ldcg(reinterpret_cast<const float2*>(p));
    lo = __ldcg(reinterpret_cast<const float2*>(p + a.stride));
  }
}

// Step 3 on a pair: right-hand sides and the Runge-Kutta combination (velocity-space terms in the parity basis,
// vlb_node.cuh).  Two lanes of one float2, so the arithmetic issues as FFMA2 / FADD2 / FMUL2 and
// shared and global accesses are 8 bytes; the two varphi taps that straddle a pair are scalar.
template <typename L, int CH, bool F0>
__device__ __forceinline__ void phase3_pair(const StageArgs<float>& a, const NodeConst<float>& nc, const float* box,
                                            const float* rows, const float* sm, PairNode& n, float2 u0_hi, float2 u0_lo,
                                            int lr, int lc, int q, int s) {
  constexpr int H = L::H, BQ = L::BQ, BS = L::BS, HS = L::HS, MS = L::MS, TQ = L::TQ;
  const float* sphi = box + NPOP * BQ * BS;
  const float* su0 = sm + L::U0_OFF;
  const float* sut = sm + L::UT_OFF;
  const float* sup = sm + L::UP_OFF;
  const float* smu = sm + L::MU_OFF;
  const int64_t stride = a.stride;
  const int bi = (lr + H) * BS + lc + HS;  // even: 8-byte aligned pairs
  const int mi = (lr + 1) * MS + lc + 2;   // even
  const int ui = lr * TS + lc;
  const float itau = a.inv_tau * a.dt;
  const float* row = rows + (lr + 1) * kRowTable;
  float rt[16];
#pragma unroll
  for (int c = 0; c < 4; ++c) reinterpret_cast<float4*>(rt)[c] = reinterpret_cast<const float4*>(row)[c];

  const float2 muN = ld2(smu + mi + MS), muS = ld2(smu + mi - MS);
  const float2 muE = make_float2(n.mu.y, smu[mi + 2]), muW = make_float2(smu[mi - 1], n.mu.x);
  // Cahn-Hilliard: M Delta mu - div(u phi) (Eq. CH), flux form with mean face values, times dt
  float2 Lp = vmul(f2(rt[E_LP]), vadd(vsub(muE, n.mu), vsub(muW, n.mu)));
  Lp = vfma(f2(rt[E_LT]), vfma(f2(rt[E_JP]), vsub(muN, n.mu), vmul(f2(rt[E_JM]), vsub(muS, n.mu))), Lp);
  float2 Ft = f2(0.0f), Fp = f2(0.0f);  // times dt
  if (CH == VLB_HYDRO) {
    const float2 upE = make_float2(n.up.y, sup[mi + 2]), upW = make_float2(sup[mi - 1], n.up.x);
    const float2 phE = make_float2(n.ph.y, sphi[bi + 2]), phW = make_float2(sphi[bi - 1], n.ph.x);
    Lp = vfma(f2(-rt[E_XN]), vmul(ld2(sut + mi + MS), ld2(sphi + bi + BS)), Lp);
    Lp = vfma(f2(rt[E_XS]), vmul(ld2(sut + mi - MS), ld2(sphi + bi - BS)), Lp);
    Lp = vfma(f2(-rt[E_YP]), vsub(vmul(upE, phE), vmul(upW, phW)), Lp);
    // n F = -phi grad mu (Eq. pbin), central differences
    const float2 pn = vmul(n.ph, n.inv);
    Ft = vmul(vmul(pn, vsub(muS, muN)), f2(a.gt * a.dt));
    Fp = vmul(vmul(pn, vsub(muW, muE)), f2(rt[E_GP]));
  }

  const int64_t gidx = (int64_t)q * a.ns + s;  // even
  if (a.dphi) {
    st2(a.dphi + gidx, Lp);  // the stabilised Cahn-Hilliard solve forms phi
  } else {
    float2 base = n.ph, base_lo = n.lo, inc = Lp;
    if (F0) {
      base = L::NU0 > NPOP ? ld2(su0 + NPOP * TQ * TS + ui) : u0_hi;
      base_lo = L::NU0 > NPOP ? ld2(su0 + (NPOP + 1) * TQ * TS + ui) : u0_lo;
      inc = vmul(f2(a.b), vadd(vadd(vsub(n.ph, base), vsub(n.lo, base_lo)), Lp));
    }
    float2 hi_o, lo_o;
    df_add(base.x, base_lo.x, inc.x, hi_o.x, lo_o.x);
    df_add(base.y, base_lo.y, inc.y, hi_o.y, lo_o.y);
    st2(a.fout + NPOP * stride + gidx, hi_o);
    st2(a.fout + (NPOP + 1) * stride + gidx, lo_o);
  }

  float2 R[NPOP];
  velocity_space(n.P, R, nc, rt, Ft, Fp, itau, a.n0, n.dn, n.ut, n.up);

  // advection, relaxation and update, two theta velocities of one magnitude (x = b: i = 3, 0; a: i = 2, 1)
  // at a time.  UW3 seen from the upwind side has the weights 1, -6, 3, 2 on the far, near, centre and
  // downwind nodes; the varphi difference keeps them whole so that its taps cancel on a uniform field.
  const float2 pv[2] = {f2(-row[E_TH + TAP_PV]), f2(-row[E_TH + 8 + TAP_PV])};
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    float t[8];
    reinterpret_cast<float4*>(t)[0] = reinterpret_cast<const float4*>(row + E_TH + 8 * x)[0];
    reinterpret_cast<float4*>(t)[1] = reinterpret_cast<const float4*>(row + E_TH + 8 * x)[1];
#pragma unroll
    for (int sgn = 0; sgn < 2; ++sgn) {
      const int i = sgn ? (x == 0 ? 0 : 1) : (x == 0 ? 3 : 2);
      const float2 tf = f2(t[sgn ? TAP_FARN : TAP_FARP]), tn = f2(t[sgn ? TAP_NEARN : TAP_NEARP]);
      const float2 td = f2(t[sgn ? TAP_DOWNN : TAP_DOWNP]), tm = f2(t[TAP_MID]);
      constexpr int STEP = BS;
      const int up = sgn ? STEP : -STEP;  // towards the upwind side
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int k = 4 * i + j;
        const float* fk = box + k * BQ * BS + bi;
        const float2 g = ld2(fk), A = ld2(fk - 2), C = ld2(fk + 2);
        float2 acc = R[k], g0 = f2(0.0f);
        if (F0) {
          g0 = ld2(su0 + k * TQ * TS + ui);
          acc = vadd(acc, vsub(g, g0));
        }
        acc = vfma(tf, ld2(fk + 2 * up), acc);
        acc = vfma(tn, ld2(fk + up), acc);
        acc = vfma(tm, g, acc);
        acc = vfma(td, ld2(fk - up), acc);
        float2 D;  // far + 3 centre - 6 near + 2 downwind along varphi
        if (j >= 2) {
          D = vfma(f2(3.0f), g, A);
          D.x = __fmaf_rn(-6.0f, A.y, D.x);
          D.y = __fmaf_rn(-6.0f, g.x, D.y);
          D.x = __fmaf_rn(2.0f, g.y, D.x);
          D.y = __fmaf_rn(2.0f, C.x, D.y);
        } else {
          D = vfma(f2(3.0f), g, C);
          D.x = __fmaf_rn(-6.0f, g.y, D.x);
          D.y = __fmaf_rn(-6.0f, C.x, D.y);
          D.x = __fmaf_rn(2.0f, A.y, D.x);
          D.y = __fmaf_rn(2.0f, g.x, D.y);
        }
        acc = vfma(pv[(j == 0 || j == 3) ? 0 : 1], D, acc);
        acc = vfma(f2(-itau), g, acc);
        st2(a.fout + k * stride + gidx, F0 ? vfma(f2(a.b), acc, g0) : vadd(acc, g));
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------------------------

// Steps 1-3 for one tile: on packed node pairs (PAIRS: the grid is known to have the chunked layout), or in scalar
// arithmetic, two or more nodes per thread (ensemble members with another layout).
template <typename L, int CH, bool F0, bool PAIRS>
__device__ __forceinline__ void tile_body(const StageArgs<float>& a, const VConst& vc, float* sm, int tid,
                                          int q0, int s0) {
  float* box = sm;
  float* co = sm + L::CO_OFF;
  pdl_wait();  // the coefficients too may come from the previous kernel (the scratch tables of vlb_step_noalloc)
  const bool pair = PAIRS || chunked<L>(a.nt, a.ns);
  if (pair)
    issue_rows<L>(a, co, q0, tid);
  else
    issue_co<L>(a, co, q0, tid);
  issue_box<L>(a, box, co, q0, s0, tid);
  cp_async_commit();
  if (F0) issue_u0<L>(a, sm + L::U0_OFF, q0, s0, tid);
  cp_async_commit();
  const int lr = tid / (TS / 2), lc = 2 * (tid % (TS / 2));  // the thread's pair of nodes
  const int q = q0 + lr, s = s0 + lc;                        // n_phi is even, so s + 1 < n_phi whenever s < n_phi
  float2 u0_hi = f2(0.0f), u0_lo = f2(0.0f);
  if (pair) load_u0_phi<L, F0>(a, q, s, u0_hi, u0_lo);
  cp_async_wait<1>();  // the box; U^n may still be in flight
  __syncthreads();
  if (pair) {
    PairNode own;
    phase2_pair<L>(a, vc.nc, box, co, sm, tid, own);
    cp_async_wait<0>();
    __syncthreads();
    pdl_trigger();
    if (q < a.nt && s < a.ns) phase3_pair<L, CH, F0>(a, vc.nc, box, co, sm, own, u0_hi, u0_lo, lr, lc, q, s);
    return;
  }
  if constexpr (PAIRS) return;
  phase2<L>(a, vc, box, co, sm, tid);
  cp_async_wait<0>();
  __syncthreads();
  pdl_trigger();
  constexpr int ROWS = L::NTH / TS;  // thread rows; each thread takes TQ / ROWS nodes of its column
#pragma unroll 1
  for (int m = 0; m < L::TQ / ROWS; ++m) {
    const int nr = tid / TS + ROWS * m, nc = tid % TS;
    if (q0 + nr < a.nt && s0 + nc < a.ns) phase3_node<L, CH, F0>(a, vc, box, co, sm, nr, nc, q0 + nr, s0 + nc);
  }
}

// Steps 1-3 for an interior tile (box inside the grid, no wrap-around) of the FP32 UW3 pair path,
// with the box and the U^n tile staged by two tensor-map copies issued by one thread and
// completing on two mbarriers.  The layout in shared memory is the one issue_box / issue_u0 produce.
// A persistent CTA (which stages many tiles) initialises the two mbarriers once and passes init =
// false with the parity of each barrier's current phase.
template <typename L, int CH, bool F0>
__device__ __forceinline__ void tile_body_tma(const StageArgs<float>& a, const VConst& vc, float* sm, int tid,
                                              int q0, int s0, const CUtensorMap* tmb, const CUtensorMap* tmu,
                                              bool init = true, unsigned ph_box = 0, unsigned ph_u0 = 0) {
  constexpr unsigned BOX_BYTES = sizeof(float) * L::NST * L::BQ * L::BS;
  constexpr unsigned U0_BYTES = sizeof(float) * L::NU0 * L::TQ * TS;
  static_assert((L::U0_OFF * sizeof(float)) % 128 == 0,
                "tensor-map destinations are 128-byte aligned");
  static_assert((L::MB_OFF * sizeof(float)) % 8 == 0, "mbarriers are 8-byte aligned");
  float* box = sm;
  float* co = sm + L::CO_OFF;
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + L::MB_OFF);
  if (init) {
    if (tid == 0) {
      mbar_init(bar, 1);
      mbar_init(bar + 1, 1);
      fence_mbar_init();
    }
    __syncthreads();
  }
  pdl_wait();
  issue_rows<L>(a, co, q0, tid);
  cp_async_commit();
  if (tid == 0) {
    mbar_expect_tx(bar, BOX_BYTES);
    tma_load_3d(box, tmb, bar, s0 - L::HS, q0 - L::H, 0);
    if (F0) {
      mbar_expect_tx(bar + 1, U0_BYTES);
      tma_load_3d(sm + L::U0_OFF, tmu, bar + 1, s0, q0, 0);
    }
    // Software pipelining through L2: the CTA that starts a.ahead tiles later (linear tile index,
    // about half a wave) will find its box and U^n tile already on chip.
    const int tiles_s = (a.ns + TS - 1) / TS;
    const int nxt = (q0 / L::TQ) * tiles_s + s0 / TS + a.ahead;
    const int qn = (nxt / tiles_s) * L::TQ, sn = (nxt % tiles_s) * TS;
    if (a.ahead > 0 && qn >= L::H && qn + L::TQ + L::H <= a.nt && sn >= L::HS && sn + TS + L::HS <= a.ns) {
      tma_prefetch_3d(tmb, sn - L::HS, qn - L::H, 0);
      if (F0) tma_prefetch_3d(tmu, sn, qn, 0);
    }
  }
  const int lr = tid / (TS / 2), lc = 2 * (tid % (TS / 2));
  float2 u0_hi = f2(0.0f), u0_lo = f2(0.0f);
  load_u0_phi<L, F0>(a, q0 + lr, s0 + lc, u0_hi, u0_lo);
  cp_async_wait<0>();
  bool ok = mbar_wait(bar, ph_box);
  if (__syncthreads_or(!ok)) {  // a copy did not land: flag it, let the copies settle, skip the tile
    if (tid == 0) {
      if (a.err) atomicExch(a.err, 2);
      mbar_wait(bar, ph_box);
      if (F0) mbar_wait(bar + 1, ph_u0);
    }
    return;
  }
  PairNode own;
  phase2_pair<L>(a, vc.nc, box, co, sm, tid, own);
  ok = F0 ? mbar_wait(bar + 1, ph_u0) : true;
  if (__syncthreads_or(!ok)) {
    if (tid == 0) {
      if (a.err) atomicExch(a.err, 2);
      mbar_wait(bar + 1, ph_u0);
    }
    return;
  }
  pdl_trigger();
  phase3_pair<L, CH, F0>(a, vc.nc, box, co, sm, own, u0_hi, u0_lo, lr, lc, q0 + lr, s0 + lc);
}

// One CTA per TQR x 32 tile, on packed node pairs.
// F0: the stage combines with U^n (stages 2 and 3); the first stage writes U_in + dt L(U_in).
// TMA: interior tiles are staged by tensor-map copies (tmb: the box of fin, tmu: the tile of f0);
// tiles whose box wraps around the grid take the per-thread copies.
template <int TQR, int CH, bool F0, bool TMA>
__global__ void __launch_bounds__(TQR*(TS / 2), TQR == 16 ? 2 : 4)
    stage_kernel(StageArgs<float> a, VConst vc, const __grid_constant__ CUtensorMap tmb,
                 const __grid_constant__ CUtensorMap tmu) {
  using L = StageLayR<TQR>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* sm = reinterpret_cast<float*>(smem_raw);
  const int q0 = blockIdx.y * L::TQ, s0 = blockIdx.x * TS;
  if constexpr (TMA) {
    if (q0 >= L::H && q0 + L::TQ + L::H <= a.nt && s0 >= L::HS && s0 + TS + L::HS <= a.ns) {
      tile_body_tma<L, CH, F0>(a, vc, sm, threadIdx.x, q0, s0, &tmb, &tmu);
      return;
    }
  }
  tile_body<L, CH, F0, true>(a, vc, sm, threadIdx.x, q0, s0);
}

// Ensemble: one launch per stage over the tiles of every member (FP32, UW3).  Block b takes work
// item items[b] = (member, tile index within the member); the member's buffers, grid and scalars
// come from its descriptor, so members of different sizes, aspect ratios and time steps share the
// launch.  TQR is the tile height chosen by the autotuner (16 or 8 rows).
// Interior tiles of members that have tensor maps (for this tile height) are staged by the bulk copies
// of tile_body_tma, and each block prefetches into L2 the work item `ahead` blocks later.
template <int TQR, int CH, bool F0>
__global__ void __launch_bounds__(TQR*(TS / 2), TQR == 16 ? 2 : 4) ensemble_stage_kernel(
                                                                       const EnsembleMember* members,
                                                                       const int2* items, int nitems, int ahead,
                                                                       int stage, int* err, VConst vc,
                                                                       const __grid_constant__ EnsembleMaps maps) {
  using L = StageLayR<TQR>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* sm = reinterpret_cast<float*>(smem_raw);
  const int2 it = items[blockIdx.x];
  const EnsembleMember& d = members[it.x];
  StageArgs<float> a;
  a.fin = d.U[stage == 0 ? 0 : stage];  // stage 0 reads U^n, 1 reads U^(1), 2 reads U^(2)
  a.f0 = F0 ? d.U[0] : nullptr;
  a.fout = d.U[stage == 2 ? 0 : stage + 1];
  a.coef = d.coef;
  a.rows = d.rows;
  a.nt = d.nt;
  a.ns = d.ns;
  a.stride = d.stride;
  a.b = stage == 0 ? 1.0f : (stage == 1 ? 0.25f : 2.0f / 3.0f);
  a.dt = d.dt;
  a.inv_tau = d.inv_tau;
  a.M = d.M;
  a.A = d.A;
  a.kappa = d.kappa;
  a.gt = d.gt;
  a.n0 = d.n0;
  a.err = err;
  a.ahead = 0;
  const int tiles_s = (d.ns + TS - 1) / TS;
  const int q0 = (it.y / tiles_s) * TQR, s0 = (it.y % tiles_s) * TS;
  if (threadIdx.x == 0 && ahead > 0 && blockIdx.x + ahead < nitems) {
    const int2 nx = items[blockIdx.x + ahead];
    const EnsembleMember& e = members[nx.x];
    const int ts = (e.ns + TS - 1) / TS, qn = (nx.y / ts) * TQR, sn = (nx.y % ts) * TS;
    if (e.maps >= 0 && qn >= L::H && qn + TQR + L::H <= e.nt && sn >= L::HS && sn + TS + L::HS <= e.ns) {
      tma_prefetch_3d(&maps.m[e.maps + stage], sn - L::HS, qn - L::H, 0);
      if (F0) tma_prefetch_3d(&maps.m[e.maps + 3], sn, qn, 0);
    }
  }
  if (d.maps >= 0 && q0 >= L::H && q0 + TQR + L::H <= d.nt && s0 >= L::HS && s0 + TS + L::HS <= d.ns) {
    tile_body_tma<L, CH, F0>(a, vc, sm, threadIdx.x, q0, s0, &maps.m[d.maps + stage], &maps.m[d.maps + 3]);
    return;
  }
  tile_body<L, CH, F0, false>(a, vc, sm, threadIdx.x, q0, s0);
}

// ---------------------------------------------------------------------------------------------
// Persistent ensemble: one cooperative launch runs whole steps.  Its CTAs (all resident at once)
// take the work items of a stage from a ticket counter and meet at a grid barrier before the next
// stage.
// The barrier is a counter and a generation word in global memory; a CTA waits for the generation
// to change for at most `budget` SM clock cycles.  On expiry it raises the ensemble's flag (2), and
// every CTA that sees the flag raised while waiting returns, so a CTA that never arrives (a lost
// CTA, or the test hook skip_cta) ends the launch with an error status instead of a hang.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_volatile_i32(const int* p) { return *reinterpret_cast<const volatile int*>(p); }
// ordering between this thread's generic-proxy accesses and later bulk (async-proxy) copies
__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;\n" ::: "memory"); }

// bar[0]: arrivals, bar[1]: generation, bar[2 + k]: the work-item tickets of stages k = 0, 1 (mod 2).
// The last CTA to arrive resets the ticket counter `reset` for the stage after the barrier before it
// releases the others.  Returns false if the barrier gave up (flag raised).
__device__ bool grid_barrier(unsigned* bar, int* err, long long budget, bool skip, int* s_ok, int reset) {
  fence_proxy_async_all();  // this thread's stores of the stage, before the next stage's bulk copies
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    const unsigned g = ld_acquire_u32(bar + 1);  // the generation cannot change before this CTA arrives
    __threadfence();                              // the CTA's stores (ordered by the CTA barrier) first
    if (!skip && atomicAdd(bar, 1u) + 1u == gridDim.x) {
      atomicExch(bar, 0u);
      atomicExch(bar + 2 + reset, 0u);
      st_release_u32(bar + 1, g + 1u);
    }
    const long long t0 = clock64();
    while (ld_acquire_u32(bar + 1) == g) {
      if (ld_volatile_i32(err) == 2) {  // another CTA gave up
        ok = 0;
        break;
      }
      if (clock64() - t0 > budget) {
        atomicCAS(err, 0, 2);
        atomicCAS(err, 1, 2);
        ok = 0;
        break;
      }
      __nanosleep(64);
    }
    fence_proxy_async_all();  // the other CTAs' stores, before this CTA's bulk copies read them
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

__device__ __forceinline__ StageArgs<float> member_args(const EnsembleMember& d, int stage, int* err) {
  StageArgs<float> a;
  a.fin = d.U[stage == 0 ? 0 : stage];  // stage 0 reads U^n, 1 reads U^(1), 2 reads U^(2)
  a.f0 = stage == 0 ? nullptr : d.U[0];
  a.fout = d.U[stage == 2 ? 0 : stage + 1];
  a.coef = d.coef;
  a.rows = d.rows;
  a.nt = d.nt;
  a.ns = d.ns;
  a.stride = d.stride;
  a.b = stage == 0 ? 1.0f : (stage == 1 ? 0.25f : 2.0f / 3.0f);
  a.dt = d.dt;
  a.inv_tau = d.inv_tau;
  a.M = d.M;
  a.A = d.A;
  a.kappa = d.kappa;
  a.gt = d.gt;
  a.n0 = d.n0;
  a.err = err;
  a.ahead = 0;
  return a;
}

// nsteps whole steps, or with only0 nsteps passes of the first stage alone (which writes only the
// scratch U^(1), so the autotuner can time it without advancing the state).
template <int TQR, int CH>
__global__ void __launch_bounds__(TQR * (TS / 2), TQR == 16 ? 2 : 4) ensemble_persistent_kernel(
    const EnsembleMember* members, const int2* items, int nitems, int nsteps, int only0, unsigned* bar, int* err,
    long long budget, int skip_cta, VConst vc, const __grid_constant__ EnsembleMaps maps) {
  using L = StageLayR<TQR>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ int s_ok;
  float* sm = reinterpret_cast<float*>(smem_raw);
  const int tid = threadIdx.x;
  if (tid == 0) {
    uint64_t* mb = reinterpret_cast<uint64_t*>(sm + L::MB_OFF);
    mbar_init(mb, 1);
    mbar_init(mb + 1, 1);
    fence_mbar_init();
  }
  __syncthreads();
  unsigned ph_box = 0, ph_u0 = 0;
  const bool skip = (int)blockIdx.x == skip_cta;
  __shared__ int s_next, s_next2;
  int gstage = 0;  // stages run so far in this launch: the ticket counter alternates between two words
  for (int n = 0; n < nsteps; ++n) {
    for (int stage = 0; stage <= (only0 ? 0 : 2); ++stage, ++gstage) {
      if (gstage > 0 && !grid_barrier(bar, err, budget, skip, &s_ok, gstage & 1)) return;
      unsigned* tickets = bar + 2 + (gstage & 1);
      // work items are handed out by a ticket counter: a CTA holds the tickets of its current and its
      // next item, so that the next item's box can be prefetched into L2 and the counter's latency
      // overlaps the current tile
      if (tid == 0) {
        s_next = (int)atomicAdd(tickets, 1u);
        s_next2 = (int)atomicAdd(tickets, 1u);
      }
      __syncthreads();
      int w = s_next, nxw = s_next2;
      while (w < nitems) {
        fence_proxy_async_all();  // the previous tile's shared-memory reads, before new copies land
        __syncthreads();          // ... and every thread has read s_next
        const int2 it = items[w];
        const EnsembleMember& d = members[it.x];
        const StageArgs<float> a = member_args(d, stage, err);
        const int tiles_s = (d.ns + TS - 1) / TS;
        const int q0 = (it.y / tiles_s) * TQR, s0 = (it.y % tiles_s) * TS;
        int after = 0;
        if (tid == 0) {
          after = (int)atomicAdd(tickets, 1u);  // used only at the end of the tile
          if (nxw < nitems) {                   // the next tile of this CTA, into L2
            const int2 nx = items[nxw];
            const EnsembleMember& e = members[nx.x];
            const int ts = (e.ns + TS - 1) / TS, qn = (nx.y / ts) * TQR, sn = (nx.y % ts) * TS;
            if (e.maps >= 0 && qn >= L::H && qn + TQR + L::H <= e.nt && sn >= L::HS && sn + TS + L::HS <= e.ns) {
              tma_prefetch_3d(&maps.m[e.maps + stage], sn - L::HS, qn - L::H, 0);
              if (stage > 0) tma_prefetch_3d(&maps.m[e.maps + 3], sn, qn, 0);
            }
          }
        }
        const bool tma = d.maps >= 0 && q0 >= L::H && q0 + TQR + L::H <= d.nt && s0 >= L::HS && s0 + TS + L::HS <= d.ns;
        if (tma) {
          if (stage == 0)
            tile_body_tma<L, CH, false>(a, vc, sm, tid, q0, s0, &maps.m[d.maps], &maps.m[d.maps + 3], false, ph_box,
                                        ph_u0);
          else
            tile_body_tma<L, CH, true>(a, vc, sm, tid, q0, s0, &maps.m[d.maps + stage], &maps.m[d.maps + 3], false,
                                       ph_box, ph_u0);
          ph_box ^= 1u;
          if (stage > 0) ph_u0 ^= 1u;
        }
        if (!tma) {
          if (stage == 0)
            tile_body<L, CH, false, false>(a, vc, sm, tid, q0, s0);
          else
            tile_body<L, CH, true, false>(a, vc, sm, tid, q0, s0);
        }
        if (tid == 0) s_next = after;
        __syncthreads();
        w = nxw;
        nxw = s_next;
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Wavefront schedule (FP32 UW3, one torus): `nsteps` whole SSP-RK3 steps in one persistent launch,
// so that the two intermediate stages of a step are consumed from L2 instead of HBM.
//
// A band is the 16 rows of one row of tiles (nb = n_theta / 16 bands, tiles_s tiles each).  Sweep
// sigma = 3 n + k (step n, stage k) visits the bands in the rotated order b = (sigma + i) mod nb,
// i = 0 .. nb - 1, and stage k of band b may run once stage k - 1 (stage 2 of step n - 1 for k = 0)
// has finished bands b - 1, b, b + 1 (the stencil reaches 2 rows, under one band).  The rotation
// makes position i of a sweep depend only on positions i .. i + 2 of the previous sweep, also across
// the periodic seam.  Band item (n, k, i) is placed in slot n nb + k lag + i, and CTAs take tiles from
// one ticket counter in slot order (stage 2 first within a slot), so that the three sweeps of a step
// trail each other by `lag` bands: the U^(1) and U^(2) a band produces is read again within about
// 2 lag bands of work, while the state U^n is read once and written once per step from HBM.
// Every dependency sits in an earlier slot when lag >= 3 and nb > 2 lag + 2, and the CTAs are all
// resident (cooperative launch), so the CTA holding the oldest unfinished ticket can always proceed.
//
// cnt[k nb + b] counts the finished tiles of stage k in band b over the launch (monotone); a wait
// polls it with acquire loads for at most `budget` SM cycles, then raises err (2) and returns, and
// every CTA that sees err == 2 while waiting returns too.  Once no reader of an intermediate band is
// left (stage 2 of band b has waited for stage 1 of b - 1 .. b + 1; stage 0 of the next step for
// stage 2 of the previous one), its lines are discarded from L2 without write-back.
// ---------------------------------------------------------------------------------------------
struct WaveMaps {
  CUtensorMap box[3];  // halo boxes of U^n, U^(1), U^(2)
  CUtensorMap tile;    // the U^n tile
};

// Band item j (0 <= j < 3 nsteps nb) in ticket order -> (n, k, i).  Slots [0, lag) hold stage 0
// only, [lag, 2 lag) stages 1, 0, [2 lag, nsteps nb) stages 2, 1, 0, then stages 2, 1 for lag
// slots and stage 2 alone for lag slots (requires nsteps nb >= 2 lag).
__host__ __device__ __forceinline__ void wave_decode(int j, int nb, int lag, int nsteps, int& n, int& k, int& i) {
  int s;
  const int steady_end = 3 * lag + 3 * (nsteps * nb - 2 * lag);
  if (j < lag) {
    s = j;
    k = 0;
  } else if (j < 3 * lag) {
    s = lag + (j - lag) / 2;
    k = 1 - (j - lag) % 2;
  } else if (j < steady_end) {
    s = 2 * lag + (j - 3 * lag) / 3;
    k = 2 - (j - 3 * lag) % 3;
  } else {
    const int jj = j - steady_end;
    if (jj < 2 * lag) {
      s = nsteps * nb + jj / 2;
      k = 2 - jj % 2;
    } else {
      s = nsteps * nb + lag + (jj - 2 * lag);
      k = 2;
    }
  }
  const int x = s - k * lag;
  n = x / nb;
  i = x - n * nb;
}

// waits until *c >= need; false if the wait gave up or another CTA did
__device__ __forceinline__ bool wave_wait(const unsigned* c, unsigned need, int* err, long long budget) {
  if (ld_acquire_u32(c) >= need) return true;
  const long long t0 = clock64();
  while (ld_acquire_u32(c) < need) {
    if (ld_volatile_i32(err) == 2) return false;
    if (clock64() - t0 > budget) {
      atomicCAS(err, 0, 2);
      atomicCAS(err, 1, 2);
      return false;
    }
    __nanosleep(32);
  }
  return true;
}

__device__ __forceinline__ void red_release_add(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}

// the 18 state arrays of one 16 x 32 tile (128-byte row segments) leave L2 without write-back
__device__ __forceinline__ void discard_tile(const float* U, int64_t stride, int ns, int q0, int s0, int tid) {
  constexpr int LINES = (NARR + 1) * 16;
  for (int l = tid; l < LINES; l += 256) {
    const int arr = l / 16, row = l % 16;
    const float* p = U + arr * stride + (int64_t)(q0 + row) * ns + s0;
    asm volatile("discard.global.L2 [%0], 128;\n" ::"l"(p) : "memory");
  }
}

template <int CH>
__global__ void __launch_bounds__(256, 2) wave_kernel(StageArgs<float> base, float* U0, float* U1, float* U2,
                                                      int nsteps, int lag, unsigned* cnt, int* err, long long budget,
                                                      int skip_cta, VConst vc,
                                                      const __grid_constant__ WaveMaps maps) {
  using L = StageLay;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ int s_item[2], s_go;
  float* sm = reinterpret_cast<float*>(smem_raw);
  const int tid = threadIdx.x;
  const int nb = base.nt / L::TQ, tiles_s = base.ns / TS;
  const int total = 3 * nsteps * nb * tiles_s;
  unsigned* tickets = cnt + 3 * nb;
  if (tid == 0) {
    uint64_t* mb = reinterpret_cast<uint64_t*>(sm + L::MB_OFF);
    mbar_init(mb, 1);
    mbar_init(mb + 1, 1);
    fence_mbar_init();
    s_item[0] = (int)atomicAdd(tickets, 1u);
    s_item[1] = (int)atomicAdd(tickets, 1u);
  }
  __syncthreads();
  unsigned ph_box = 0, ph_u0 = 0;
  int t = s_item[0], tn = s_item[1];
  while (t < total) {
    const int j = t / tiles_s, c = t - j * tiles_s;
    int n, k, i;
    wave_decode(j, nb, lag, nsteps, n, k, i);
    const int b = (3 * n + k + i) % nb;
    const int q0 = b * L::TQ, s0 = c * TS;
    if (tid == 0) {
      // dependencies: the previous sweep on bands b - 1, b, b + 1
      bool ok = true;
      const int kp = k == 0 ? 2 : k - 1;
      const unsigned need = (unsigned)((k == 0 ? n : n + 1) * tiles_s);
      if (k > 0 || n > 0) {
        for (int d = -1; d <= 1 && ok; ++d) ok = wave_wait(cnt + kp * nb + (b + d + nb) % nb, need, err, budget);
      }
      fence_proxy_async_all();  // the other CTAs' stores, before this CTA's bulk copies read them
      // the next tile of this CTA, into L2 (a hint: its inputs may not be final yet)
      if (ok && tn < total) {
        const int jn = tn / tiles_s, cn = tn - jn * tiles_s;
        int nn, kn, in_;
        wave_decode(jn, nb, lag, nsteps, nn, kn, in_);
        const int qn = ((3 * nn + kn + in_) % nb) * L::TQ, sn = cn * TS;
        if (qn >= L::H && qn + L::TQ + L::H <= base.nt && sn >= L::HS && sn + TS + L::HS <= base.ns) {
          tma_prefetch_3d(&maps.box[kn], sn - L::HS, qn - L::H, 0);
          if (kn > 0) tma_prefetch_3d(&maps.tile, sn, qn, 0);
        }
      }
      s_go = ok;
      s_item[0] = (int)atomicAdd(tickets, 1u);  // the ticket after next, used at the end of the tile
    }
    __syncthreads();
    if (!s_go) return;
    // no reader of these intermediate bands is left
    if (k == 2) discard_tile(U1, base.stride, base.ns, q0, s0, tid);
    if (k == 0 && n > 0) discard_tile(U2, base.stride, base.ns, q0, s0, tid);
    StageArgs<float> a = base;
    a.fin = k == 0 ? U0 : (k == 1 ? U1 : U2);
    a.f0 = k == 0 ? nullptr : U0;
    a.fout = k == 0 ? U1 : (k == 1 ? U2 : U0);
    a.b = k == 0 ? 1.0f : (k == 1 ? 0.25f : 2.0f / 3.0f);
    a.ahead = 0;
    a.err = err;
    const bool tma = q0 >= L::H && q0 + L::TQ + L::H <= a.nt && s0 >= L::HS && s0 + TS + L::HS <= a.ns;
    if (tma) {
      if (k == 0)
        tile_body_tma<L, CH, false>(a, vc, sm, tid, q0, s0, &maps.box[0], &maps.tile, false, ph_box, ph_u0);
      else
        tile_body_tma<L, CH, true>(a, vc, sm, tid, q0, s0, &maps.box[k], &maps.tile, false, ph_box, ph_u0);
      ph_box ^= 1u;
      if (k > 0) ph_u0 ^= 1u;
    } else {
      if (k == 0)
        tile_body<L, CH, false, true>(a, vc, sm, tid, q0, s0);
      else
        tile_body<L, CH, true, true>(a, vc, sm, tid, q0, s0);
    }
    // this tile's stores, before the consumers' bulk copies; the CTA's shared-memory reads, before
    // the next tile's copies land
    fence_proxy_async_all();
    __syncthreads();
    if (ld_volatile_i32(err) == 2) return;  // a copy of this CTA (or another) gave up
    if (tid == 0 && (int)blockIdx.x != skip_cta) {  // skip_cta: test hook, a CTA that never reports
      __threadfence();
      red_release_add(cnt + k * nb + b, 1u);
    }
    t = tn;
    tn = s_item[0];
    __syncthreads();  // every thread has read s_item before thread 0 rewrites it
  }
}

VConst make_vconst() {
  const VelocityConsts d = velocity_consts();
  VConst c;
  c.nc = make_node_const<float>();
  for (int i = 0; i < 4; ++i) {
    c.v[i] = (float)d.v[i];
    c.w[i] = (float)d.w[i];
    for (int m = 0; m < 4; ++m) {
      c.K[i][m] = (float)d.K[i][m];
      c.ww[i][m] = (float)(d.w[i] * d.w[m]);
    }
  }
  return c;
}

// Tile height of a solver's stage launches.  8-row tiles take 56 KB and 128 threads, so four share an SM (16
// warps, as two 16-row tiles) with finer-grained overlap of copies and arithmetic: us per step with 16 / 8
// rows 22.6 / 21.3 (256 x 512), 45.2 / 37.5 (400 x 800), 69.7 / 57.9 (512 x 1024), 218.5 / 203.6 (1024 x 2048); small
// grids too, where each SM holds at most one tile (64 x 128: 13.7 / 10.3).  In between, where one 16-row tile per SM
// holds the grid but one 8-row tile does not, the second 8-row tile of an SM costs more than it saves (192 x 384:
// 15.0 / 17.2, 256 x 256: 14.5 / 16.3).  4-row tiles are no better than 8 above 64 x 128.  Grids with more 8-row
// tiles along theta than a grid dimension holds take 16 rows too (vlb_create admits 65535 x 16 rows).
constexpr int kSms = 152, kGridRows = 65535;
int stage_rows_rule(int nt, int ns) {
  const int64_t cols = (ns + TS - 1) / TS, t8 = cols * ((nt + 7) / 8), t16 = cols * ((nt + 15) / 16);
  if ((nt + 7) / 8 > kGridRows) return 16;
  return t8 > kSms && t16 <= kSms ? 16 : 8;
}

// Per-device, per-kernel one-time set-up (dynamic shared memory opt-in).
template <typename K>
cudaError_t ensure_smem(K kernel, size_t bytes, int& mask) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 32 && (mask & (1 << dev))) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess && dev < 32) mask |= (1 << dev);
  return e;
}

template <int TQR, int CH, bool F0, bool TMA>
cudaError_t launch_pairs(const StageArgs<float>& a, cudaStream_t st, const StageMaps* maps) {
  using L = StageLayR<TQR>;
  static int mask = 0;
  cudaError_t e = ensure_smem(stage_kernel<TQR, CH, F0, TMA>, L::BYTES, mask);
  if (e != cudaSuccess) return e;
  static const VConst vc = make_vconst();
  static const StageMaps none = {};
  const StageMaps& m = maps ? *maps : none;
  StageArgs<float> args = a;
  args.ahead = 0;
  if (TMA) {
    static int resident[32] = {0};  // CTAs of this kernel resident at once, per device
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if (dev < 32 && resident[dev] == 0) {
      int per_sm = 0, sms = 0;
      if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, stage_kernel<TQR, CH, F0, TMA>, L::NTH,
                                                             L::BYTES)) != cudaSuccess)
        return e;
      if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
      resident[dev] = per_sm * sms;
    }
    // half a wave ahead (about the next tile started on the same SM) measured best on GB300 (16-row tiles): 0.217 ms
    // per step on 1024 x 2048 against 0.225 (one wave), 0.221 (a quarter) and 0.234 (no prefetch)
    args.ahead = dev < 32 ? resident[dev] / 2 : 0;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((a.ns + TS - 1) / TS, (a.nt + L::TQ - 1) / L::TQ);
  cfg.blockDim = dim3(L::NTH);
  cfg.dynamicSmemBytes = L::BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, stage_kernel<TQR, CH, F0, TMA>, args, vc, m.box, m.tile);
}

template <int TQR, int CH, bool F0>
cudaError_t launch_ens(const EnsembleMember* members, const int2* items, int nitems, int stage, int* err,
                       cudaStream_t st, const EnsembleMaps& maps) {
  using L = StageLayR<TQR>;
  static int mask = 0;
  cudaError_t e = ensure_smem(ensemble_stage_kernel<TQR, CH, F0>, L::BYTES, mask);
  if (e != cudaSuccess) return e;
  static const VConst vc = make_vconst();
  static int resident[32] = {0};  // blocks of this kernel resident at once, per device
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev < 32 && resident[dev] == 0) {
    int per_sm = 0, sms = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ensemble_stage_kernel<TQR, CH, F0>, L::NTH,
                                                           L::BYTES)) != cudaSuccess)
      return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    resident[dev] = per_sm * sms;
  }
  const int ahead = dev < 32 ? resident[dev] / 2 : 0;  // half a wave, as for a single torus
  ensemble_stage_kernel<TQR, CH, F0><<<nitems, L::NTH, L::BYTES, st>>>(members, items, nitems, ahead, stage, err, vc,
                                                                     maps);
  return cudaGetLastError();
}

template <int TQR, int CH>
cudaError_t launch_pers(const EnsembleMember* members, const int2* items, int nitems, int nsteps, int only0,
                        unsigned* bar, int* err, long long budget, int skip_cta, int ctas_per_sm, cudaStream_t st,
                        const EnsembleMaps& maps, int* grid_out) {
  using L = StageLayR<TQR>;
  static int mask = 0;
  cudaError_t e = ensure_smem(ensemble_persistent_kernel<TQR, CH>, L::BYTES, mask);
  if (e != cudaSuccess) return e;
  static const VConst vc = make_vconst();
  static int occ[32] = {0}, sms[32] = {0};
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev >= 32) return cudaErrorInvalidDevice;
  if (occ[dev] == 0) {
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[dev], ensemble_persistent_kernel<TQR, CH>, L::NTH,
                                                           L::BYTES)) != cudaSuccess)
      return e;
    if ((e = cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if (occ[dev] < 1) return cudaErrorInvalidConfiguration;
  }
  const int per_sm = ctas_per_sm > 0 && ctas_per_sm < occ[dev] ? ctas_per_sm : occ[dev];
  int grid = per_sm * sms[dev];
  if (grid > nitems) grid = nitems;
  if (grid_out) *grid_out = grid;
  if (grid < 1 || nsteps < 1) return cudaSuccess;
  // the arrival counter and both ticket counters start at zero (a launch that gave up may have left
  // arrivals or tickets behind); the generation word keeps counting
  if ((e = cudaMemsetAsync(bar, 0, sizeof(unsigned), st)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(bar + 2, 0, 2 * sizeof(unsigned), st)) != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(L::NTH);
  cfg.dynamicSmemBytes = L::BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // all CTAs resident at once: the grid barrier is safe
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, ensemble_persistent_kernel<TQR, CH>, members, items, nitems, nsteps, only0, bar, err,
                            budget, skip_cta, vc, maps);
}

template <int TQR>
cudaError_t launch_ens_rows(const EnsembleMember* members, const int2* items, int nitems, int stage, int ch_mode,
                            int* err, cudaStream_t st, const EnsembleMaps& maps) {
  if (ch_mode == VLB_HYDRO)
    return stage == 0 ? launch_ens<TQR, VLB_HYDRO, false>(members, items, nitems, stage, err, st, maps)
                      : launch_ens<TQR, VLB_HYDRO, true>(members, items, nitems, stage, err, st, maps);
  return stage == 0 ? launch_ens<TQR, VLB_DIFFUSIVE, false>(members, items, nitems, stage, err, st, maps)
                    : launch_ens<TQR, VLB_DIFFUSIVE, true>(members, items, nitems, stage, err, st, maps);
}


template <int TQR, int CH>
cudaError_t launch_rows(const StageArgs<float>& a, cudaStream_t st, const StageMaps* maps) {
  if (maps)
    return a.f0 ? launch_pairs<TQR, CH, true, true>(a, st, maps) : launch_pairs<TQR, CH, false, true>(a, st, maps);
  return a.f0 ? launch_pairs<TQR, CH, true, false>(a, st, nullptr) : launch_pairs<TQR, CH, false, false>(a, st, nullptr);
}

template <typename T, int ADV, int CH>
cudaError_t launch_one(const StageArgs<T>& a, cudaStream_t st, const StageMaps* maps) {
  if constexpr (sizeof(T) == 4 && ADV == VLB_UW3) {
    if (chunked<StageLay>(a.nt, a.ns)) {  // n_phi % 4 == 0: packed node pairs
      const int rows = stage_rows(a.nt, a.ns);
      return rows == 16 ? launch_rows<16, CH>(a, st, maps) : launch_rows<8, CH>(a, st, maps);
    }
  }
  return launch_direct<T>(a, ADV, CH, st);  // FP64, WENO5, and FP32 off the packed layout (vlb_direct.cu)
}

using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encoder() {
  static EncodeTiled fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiled>(p);
  }
  return fn;
}

// 3-D map over the 18 FP32 state arrays: (varphi, theta, array), box bx x by x arrays.
cudaError_t encode_state_map(CUtensorMap* m, const float* base, int nt, int ns, int64_t stride, int bx, int by,
                             int arrays) {
  EncodeTiled fn = encoder();
  if (!fn) return cudaErrorNotSupported;
  const cuuint64_t dims[3] = {(cuuint64_t)ns, (cuuint64_t)nt, (cuuint64_t)(NARR + 1)};
  const cuuint64_t strides[2] = {(cuuint64_t)ns * sizeof(float), (cuuint64_t)stride * sizeof(float)};
  const cuuint32_t box[3] = {(cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)arrays};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

int stage_rows(int nt, int ns) { return stage_rows_rule(nt, ns); }

bool stage_maps_apply(int nt, int ns) { return chunked<StageLay>(nt, ns); }

cudaError_t make_stage_maps(const float* fin, const float* f0, int nt, int ns, int64_t stride, int rows,
                            StageMaps* out) {
  using L = StageLay;
  if (!stage_maps_apply(nt, ns) || stride % 4 != 0 || ((uintptr_t)fin) % 16 != 0 || ((uintptr_t)f0) % 16 != 0)
    return cudaErrorInvalidValue;
  cudaError_t e = encode_state_map(&out->box, fin, nt, ns, stride, L::BS, rows + 2 * L::H, L::NST);
  if (e == cudaSuccess) e = encode_state_map(&out->tile, f0, nt, ns, stride, TS, rows, rows == 16 ? StageLayR<16>::NU0 : StageLayR<8>::NU0);
  return e;
}

template <typename T>
cudaError_t launch_stage(const StageArgs<T>& a, int advection, int ch_mode, cudaStream_t s, const StageMaps* maps) {
  if (advection == VLB_UW3)
    return ch_mode == VLB_HYDRO ? launch_one<T, VLB_UW3, VLB_HYDRO>(a, s, maps)
                                : launch_one<T, VLB_UW3, VLB_DIFFUSIVE>(a, s, maps);
  return ch_mode == VLB_HYDRO ? launch_one<T, VLB_WENO5, VLB_HYDRO>(a, s, nullptr)
                              : launch_one<T, VLB_WENO5, VLB_DIFFUSIVE>(a, s, nullptr);
}

cudaError_t launch_ensemble_stage(const EnsembleMember* members, const int2* items, int nitems, int stage,
                                  int tile_rows, int ch_mode, int* err, cudaStream_t s, const EnsembleMaps* maps) {
  if (nitems <= 0) return cudaSuccess;
  static const EnsembleMaps none = {};
  const EnsembleMaps& m = maps ? *maps : none;
  if (tile_rows == 8) return launch_ens_rows<8>(members, items, nitems, stage, ch_mode, err, s, m);
  return launch_ens_rows<16>(members, items, nitems, stage, ch_mode, err, s, m);
}

cudaError_t launch_ensemble_persistent(const EnsembleMember* members, const int2* items, int nitems, int nsteps,
                                       int only0, int tile_rows, int ch_mode, unsigned* bar, int* err, long long budget,
                                       int skip_cta, int ctas_per_sm, cudaStream_t s, const EnsembleMaps* maps,
                                       int* grid_out) {
  if (nitems <= 0) return cudaSuccess;
  static const EnsembleMaps none = {};
  const EnsembleMaps& m = maps ? *maps : none;
  if (tile_rows == 8)
    return ch_mode == VLB_HYDRO ? launch_pers<8, VLB_HYDRO>(members, items, nitems, nsteps, only0, bar, err, budget,
                                                             skip_cta, ctas_per_sm, s, m, grid_out)
                                : launch_pers<8, VLB_DIFFUSIVE>(members, items, nitems, nsteps, only0, bar, err, budget,
                                                                 skip_cta, ctas_per_sm, s, m, grid_out);
  return ch_mode == VLB_HYDRO ? launch_pers<16, VLB_HYDRO>(members, items, nitems, nsteps, only0, bar, err, budget,
                                                            skip_cta, ctas_per_sm, s, m, grid_out)
                              : launch_pers<16, VLB_DIFFUSIVE>(members, items, nitems, nsteps, only0, bar, err, budget,
                                                                skip_cta, ctas_per_sm, s, m, grid_out);
}

bool wave_schedule_ok(int nb, int lag, int nsteps) {
  if (lag < 3 || nb <= 2 * lag + 2 || nsteps < 1) return false;
  // every band item's dependencies sit in earlier tickets (checked by enumeration for small launches)
  if ((int64_t)3 * nsteps * nb > (int64_t)1 << 20) return true;
  std::vector<int> pos((size_t)3 * nsteps * nb, -1);  // ticket position of (n, k, band)
  for (int j = 0; j < 3 * nsteps * nb; ++j) {
    int n, k, i;
    wave_decode(j, nb, lag, nsteps, n, k, i);
    if (n < 0 || n >= nsteps || k < 0 || k > 2 || i < 0 || i >= nb) return false;
    const size_t at = ((size_t)n * 3 + k) * nb + (3 * n + k + i) % nb;
    if (pos[at] != -1) return false;  // each band item exactly once
    pos[at] = j;
  }
  for (int n = 0; n < nsteps; ++n)
    for (int k = 0; k < 3; ++k)
      for (int b = 0; b < nb; ++b) {
        if (k == 0 && n == 0) continue;
        const int np = k == 0 ? n - 1 : n, kp = k == 0 ? 2 : k - 1;
        for (int d = -1; d <= 1; ++d)
          if (pos[((size_t)np * 3 + kp) * nb + (b + d + nb) % nb] >= pos[((size_t)n * 3 + k) * nb + b]) return false;
      }
  return true;
}

bool wave_apply(int nt, int ns) {
  using L = StageLay;
  return stage_maps_apply(nt, ns) && nt % L::TQ == 0 && ns % TS == 0 && nt / L::TQ > 2 * kWaveLag + 2;
}

int wave_counter_words(int nt) { return 3 * (nt / 16) + 1; }

template <int CH>
cudaError_t launch_wave_t(const StageArgs<float>& a, float* U0, float* U1, float* U2, int nsteps, unsigned* cnt,
                          long long budget, int skip_cta, cudaStream_t st, const WaveMaps& maps, int* grid_out) {
  using L = StageLay;
  static int mask = 0;
  cudaError_t e = ensure_smem(wave_kernel<CH>, L::BYTES, mask);
  if (e != cudaSuccess) return e;
  static const VConst vc = make_vconst();
  static int occ[32] = {0}, sms[32] = {0};
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev >= 32) return cudaErrorInvalidDevice;
  if (occ[dev] == 0) {
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[dev], wave_kernel<CH>, 256, L::BYTES)) != cudaSuccess)
      return e;
    if ((e = cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if (occ[dev] < 1) return cudaErrorInvalidConfiguration;
  }
  const int nb = a.nt / L::TQ, tiles = nb * (a.ns / TS);
  int grid = occ[dev] * sms[dev];
  if (grid > 3 * tiles) grid = 3 * tiles;
  if (grid_out) *grid_out = grid;
  if ((e = cudaMemsetAsync(cnt, 0, sizeof(unsigned) * wave_counter_words(a.nt), st)) != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = L::BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // every ticket holder is resident: the waits end
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, wave_kernel<CH>, a, U0, U1, U2, nsteps, kWaveLag, cnt, a.err, budget, skip_cta, vc,
                            maps);
}

cudaError_t launch_wave(const StageArgs<float>& a, int ch_mode, float* U0, float* U1, float* U2, int nsteps,
                        unsigned* cnt, long long budget, int skip_cta, cudaStream_t st, const StageMaps* stage_maps,
                        int* grid_out) {
  if (!wave_apply(a.nt, a.ns) || !stage_maps || nsteps < 1 || nsteps > kWaveMaxSteps) return cudaErrorInvalidValue;
  for (float* u : {U0, U1, U2})
    if (((uintptr_t)u) % 128 != 0 || a.stride % 32 != 0) return cudaErrorInvalidValue;  // discarded lines
  WaveMaps m;
  m.box[0] = stage_maps[0].box;
  m.box[1] = stage_maps[1].box;
  m.box[2] = stage_maps[2].box;
  m.tile = stage_maps[1].tile;
  return ch_mode == VLB_HYDRO
             ? launch_wave_t<VLB_HYDRO>(a, U0, U1, U2, nsteps, cnt, budget, skip_cta, st, m, grid_out)
             : launch_wave_t<VLB_DIFFUSIVE>(a, U0, U1, U2, nsteps, cnt, budget, skip_cta, st, m, grid_out);
}

template cudaError_t launch_stage<float>(const StageArgs<float>&, int, int, cudaStream_t, const StageMaps*);
template cudaError_t launch_stage<double>(const StageArgs<double>&, int, int, cudaStream_t, const StageMaps*);

}  // namespace vlb
