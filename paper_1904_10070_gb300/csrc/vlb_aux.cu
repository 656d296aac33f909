// Initialisation, state conversion, field read-out and FP64 diagnostic reductions.
//
// These kernels run once per set/get call or once per diagnostic, not per time step.  Their
// arithmetic is done in FP64 (the FP32 state is widened on load; its totals in float pairs), so the read-outs
// and the conserved totals carry no FP32 rounding beyond that of the state itself.
#include <math.h>

#include "vlb_node.cuh"

namespace vlb {

namespace {

constexpr int TOTAL_BLOCKS = 512;
constexpr int TOTAL_THREADS = 256;
constexpr int NSUM = 8;

struct VD {
  double v[4], w[4];
};

VD make_vd() {
  const VelocityConsts c = velocity_consts();
  VD d;
  for (int i = 0; i < 4; ++i) {
    d.v[i] = c.v[i];
    d.w[i] = c.w[i];
  }
  return d;
}

__device__ __forceinline__ int wrapi(int x, int n) {
  x %= n;
  return x < 0 ? x + n : x;
}

// phi as stored: one array in FP64 mode, hi + lo in FP32 mode.
template <typename T>
__device__ __forceinline__ void store_phi(T* state, int64_t stride, int64_t idx, double v) {
  const T hi = (T)v;
  state[NPOP * stride + idx] = hi;
  if (sizeof(T) == 4) state[(NPOP + 1) * stride + idx] = (T)(v - (double)hi);
}

template <typename T>
__device__ __forceinline__ double load_phi(const T* state, int64_t stride, int64_t idx) {
  double v = (double)state[NPOP * stride + idx];
  if (sizeof(T) == 4) v += (double)state[(NPOP + 1) * stride + idx];
  return v;
}

// f := f^eq(rho, u) (Eq. feq), phi := phi, stored as the deviation g = f^eq - n0 w_i w_j
// = w_i w_j ((n - n0) + n (poly - 1)).  FP64 state: evaluated in FP64.  FP32 state: n - n0 is formed in
// FP64 (exact enough that its rounding to FP32 is the only error), the Hermite polynomial and the
// product in FP32 -- every term is small next to the stored value's own rounding -- so the
// initialisation does not run on GB300's FP64 units.
template <typename T>
__global__ void init_feq_kernel(T* state, int64_t stride, const double* rho, const double* ut, const double* up,
                                const double* phi, int64_t n, double n0, VD vd) {
  using C = T;  // arithmetic of the polynomial: the state precision
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n; idx += (int64_t)gridDim.x * blockDim.x) {
    const double nn = rho[idx];
    const C a = (C)ut[idx], b = (C)up[idx], dn = (C)(nn - n0), nc = (C)nn;
    const C usq = a * a + b * b;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const C xi = (C)vd.v[i] * a + (C)vd.v[j] * b;
        const C pm1 = xi + C(0.5) * (xi * xi - usq) + xi * (xi * xi - C(3) * usq) * C(1.0 / 6.0);
        state[(4 * i + j) * stride + idx] = (T)((C)(vd.w[i] * vd.w[j]) * (dn + nc * pm1));
      }
    store_phi(state, stride, idx, phi[idx]);
  }
}

__device__ __forceinline__ double ref_pop(int k, double n0, const VD& vd) {
  return k < NPOP ? n0 * vd.w[k >> 2] * vd.w[k & 3] : 0.0;
}

template <typename T>
__global__ void convert_in_kernel(T* state, int64_t stride, const double* src, int64_t n, double n0, VD vd) {
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n * NARR;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = idx / n, i = idx - k * n;
    if (k == NPOP)
      store_phi(state, stride, i, src[idx]);
    else
      state[k * stride + i] = (T)(src[idx] - ref_pop((int)k, n0, vd));
  }
}

template <typename T>
__global__ void convert_out_kernel(double* dst, const T* state, int64_t stride, int64_t n, double n0, VD vd) {
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n * NARR;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = idx / n, i = idx - k * n;
    dst[idx] = k == NPOP ? load_phi(state, stride, i) : (double)state[k * stride + i] + ref_pop((int)k, n0, vd);
  }
}

template <typename T>
__device__ __forceinline__ void node_moments(const T* state, int64_t stride, int64_t idx, const VD& vd, double n0,
                                             double& n, double& ut, double& up) {
  double row[4] = {0, 0, 0, 0}, col[4] = {0, 0, 0, 0};
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double x = (double)state[(4 * i + j) * stride + idx];
      row[i] += x;
      col[j] += x;
    }
  n = n0 + ((row[0] + row[1]) + (row[2] + row[3]));
  const double inv_n = 1.0 / n;  // one FP64 division per node
  ut = (vd.v[0] * row[0] + vd.v[1] * row[1] + vd.v[2] * row[2] + vd.v[3] * row[3]) * inv_n;
  up = (vd.v[0] * col[0] + vd.v[1] * col[1] + vd.v[2] * col[2] + vd.v[3] * col[3]) * inv_n;
}

// rho, u (Sec. 2.3 moments), phi and mu (Eq. mu) in FP64; one CTA row per theta row (blockIdx.y).
template <typename T>
__global__ void fields_kernel(const T* state, int64_t stride, const double* coefd, int nt, int ns, double A,
                              double kappa, double n0, double* rho, double* ut, double* up, double* phi, double* mu, VD vd) {
  const int q = blockIdx.y, s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= ns) return;
  const int64_t idx = (int64_t)q * ns + s;
  double nn, a, b;
  node_moments(state, stride, idx, vd, n0, nn, a, b);
  rho[idx] = nn;
  ut[idx] = a;
  up[idx] = b;
  const int qn = q + 1 == nt ? 0 : q + 1, qs = q == 0 ? nt - 1 : q - 1;
  const int se = s + 1 == ns ? 0 : s + 1, sw = s == 0 ? ns - 1 : s - 1;
  const double p0 = load_phi(state, stride, idx);
  const double pn = load_phi(state, stride, (int64_t)qn * ns + s);
  const double ps = load_phi(state, stride, (int64_t)qs * ns + s);
  const double pe = load_phi(state, stride, (int64_t)q * ns + se);
  const double pw = load_phi(state, stride, (int64_t)q * ns + sw);
  const double lap = coefd[C_LT * nt + q] * (coefd[C_JP * nt + q] * (pn - p0) - coefd[C_JM * nt + q] * (p0 - ps)) +
                     coefd[C_LP * nt + q] * (pe - 2.0 * p0 + pw);
  phi[idx] = p0;
  mu[idx] = -A * p0 * (1.0 - p0 * p0) - kappa * lap;
}

// Per-block FP64 sums: mass, phi total, Psi (Eq. Landau), max |u|, non-finite count (NTOT of a block's NSUM slots).
// Warp, then block reduction in a fixed order.
constexpr int NTOT = 5;
__device__ __forceinline__ void reduce_totals(double (&acc)[NSUM], double* partials) {
  __shared__ double red[TOTAL_THREADS / 32][NSUM];
#pragma unroll
  for (int k = 0; k < NTOT; ++k) {
    double x = acc[k];
    for (int o = 16; o > 0; o >>= 1) {
      const double y = __shfl_down_sync(0xffffffffu, x, o);
      x = (k == 3) ? fmax(x, y) : x + y;
    }
    acc[k] = x;
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0)
    for (int k = 0; k < NSUM; ++k) red[wid][k] = acc[k];
  __syncthreads();
  if (threadIdx.x < NTOT) {
    const int k = threadIdx.x;
    double x = 0.0;
    for (int w = 0; w < TOTAL_THREADS / 32; ++w) x = (k == 3) ? fmax(x, red[w][k]) : x + red[w][k];
    partials[blockIdx.x * NSUM + k] = x;
  }
}

// One node's share of the totals in FP64; acc[3] collects |u|^2 (the root is taken once, after the maximum:
// a correctly rounded root is monotone).
template <typename T>
__device__ __forceinline__ void node_totals(const T* state, int64_t stride, const double* coefd, int nt, int ns, int q,
                                            int s, double A, double kappa, double n0, double gt, const VD& vd,
                                            double (&acc)[NSUM]) {
  const int64_t idx = (int64_t)q * ns + s;
  double nn, a, b;
  node_moments(state, stride, idx, vd, n0, nn, a, b);
  const double dA = coefd[C_DA * nt + q];
  const double p0 = load_phi(state, stride, idx);
  const double pn = load_phi(state, stride, (int64_t)wrapi(q + 1, nt) * ns + s);
  const double ps = load_phi(state, stride, (int64_t)wrapi(q - 1, nt) * ns + s);
  const double pe = load_phi(state, stride, (int64_t)q * ns + wrapi(s + 1, ns));
  const double pw = load_phi(state, stride, (int64_t)q * ns + wrapi(s - 1, ns));
  const double g1 = (pn - ps) * gt, g2 = (pe - pw) * coefd[C_GP * nt + q];
  const double om = 1.0 - p0 * p0;
  acc[0] += nn * dA;
  acc[1] += p0 * dA;
  acc[2] += (0.25 * A * om * om + 0.5 * kappa * (g1 * g1 + g2 * g2)) * dA;
  const double u2 = a * a + b * b;
  acc[3] = fmax(acc[3], u2);
  if (!isfinite(nn) || !isfinite(u2) || !isfinite(p0)) acc[4] += 1.0;
}

template <typename T>
__global__ void __launch_bounds__(TOTAL_THREADS) totals_kernel(const T* state, int64_t stride, const double* coefd,
                                                               int nt, int ns, double A, double kappa, double n0,
                                                               double gt, double* partials, VD vd) {
  const int64_t n = (int64_t)nt * ns;
  double acc[NSUM] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n; idx += (int64_t)gridDim.x * blockDim.x) {
    const int q = (int)(idx / ns);
    node_totals(state, stride, coefd, nt, ns, q, (int)(idx - (int64_t)q * ns), A, kappa, n0, gt, vd, acc);
  }
  acc[3] = sqrt(acc[3]);
  reduce_totals(acc, partials);
}

// ---- Totals of an FP32 state in float pairs -----------------------------------------------------------
// The FP64 units (one warp instruction per 19 cycles and SM) made the totals of 1024 x 2048 cost 558 us at
// about 100 FP64 operations a node.  Here a node's quantities are unevaluated pairs h + l of floats with error-free
// sums and products (Dekker 1971, Knuth), 2^-46 relative each, and FP64 takes over at the row.  What a sum over
// many nodes averages out may stay at that; what it does not is done as exactly as in FP64: differences keep their
// relative accuracy (diff, 1 - phi^2 as a product), phi is summed with the rounding of its low words carried, and
// the node of the largest |u| is evaluated again in FP64.  About 560 FP32 operations a node, 100 us (86 with pairs
// alone).  A node whose values leave the range in which the pairs neither overflow nor lose bits to underflow takes the
// FP64 path.
struct FF {
  float h, l;
};
__device__ __forceinline__ FF quick_sum(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ FF two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ FF operator+(FF a, FF b) {
  const FF s = two_sum(a.h, b.h);
  return quick_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ FF operator-(FF a) { return {-a.h, -a.l}; }
__device__ __forceinline__ FF operator-(FF a, FF b) { return a + (-b); }
// a - b, accurate relative to the difference
__device__ __forceinline__ FF diff(FF a, FF b) {
  const FF s = two_sum(a.h, -b.h), t = two_sum(a.l, -b.l), r = quick_sum(s.h, __fadd_rn(s.l, t.h));
  return quick_sum(r.h, __fadd_rn(r.l, t.l));
}
__device__ __forceinline__ bool exceeds(FF a, FF b) { return a.h > b.h || (a.h == b.h && a.l > b.l); }
__device__ __forceinline__ FF operator*(FF a, FF b) {
  const float p = __fmul_rn(a.h, b.h);
  return quick_sum(p, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ FF operator/(FF a, FF b) {
  const float q = __fdiv_rn(a.h, b.h);
  const FF p = b * FF{q, 0.0f}, r = a - p;
  return quick_sum(q, __fdiv_rn(r.h, b.h));
}
__device__ __forceinline__ FF to_ff(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ double to_d(FF a) { return (double)a.h + (double)a.l; }

// W threads (a power of two) share a segment of `len` nodes of a row; `segs` segments a row.
__global__ void __launch_bounds__(TOTAL_THREADS) totals32_kernel(const float* state, int64_t stride,
                                                                 const double* coefd, int nt, int ns, int W, int segs,
                                                                 int len, double A, double kappa, double n0, double gt,
                                                                 double* partials, VD vd) {
  const int c = threadIdx.x & (W - 1), rb = TOTAL_THREADS / W;
  const FF va = to_ff(vd.v[2]), vb = to_ff(vd.v[3]), gtf = to_ff(gt), A4 = to_ff(0.25 * A), k2 = to_ff(0.5 * kappa);
  const FF n0f = to_ff(n0), one = {1.0f, 0.0f};
  const float *hi = state + NPOP * stride, *lo = hi + stride;
  double acc[NSUM] = {0, 0, 0, 0, 0, 0, 0, 0};
  FF best = {0.0f, 0.0f};  // largest |u|^2, and its node
  int64_t best_at = -1;
  for (int64_t unit = blockIdx.x * (int64_t)rb + threadIdx.x / W; unit < (int64_t)nt * segs;
       unit += (int64_t)gridDim.x * rb) {
    const int q = (int)(unit / segs), first = (int)(unit - (int64_t)q * segs) * len;
    const int last = first + len < ns ? first + len : ns;
    const int64_t rn = (int64_t)(q + 1 < nt ? q + 1 : 0) * ns, rs = (int64_t)(q > 0 ? q - 1 : nt - 1) * ns;
    const int64_t r0 = (int64_t)q * ns;
    const FF gp = to_ff(coefd[C_GP * nt + q]);
    FF m = {0.0f, 0.0f}, ph = m, psi = m;
    float ph3 = 0.0f;  // rounding of ph's low word
    int count = 0;
    for (int s = first + c; s < last; s += W) {
      const int se = s + 1 < ns ? s + 1 : 0, sw = s > 0 ? s - 1 : ns - 1;
      const float* f = state + r0 + s;
      FF S[4], OB = {0.0f, 0.0f}, OA = OB;
      float big = 0.0f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float g0 = f[(4 * i) * stride], g1 = f[(4 * i + 1) * stride];
        const float g2 = f[(4 * i + 2) * stride], g3 = f[(4 * i + 3) * stride];
        big = fmaxf(fmaxf(big, fmaxf(fabsf(g0), fabsf(g1))), fmaxf(fabsf(g2), fabsf(g3)));
        S[i] = two_sum(g3, g0) + two_sum(g2, g1);
        OB = OB + two_sum(g3, -g0);
        OA = OA + two_sum(g2, -g1);
      }
      const FF p0 = {hi[r0 + s], lo[r0 + s]};
      const FF pn = {hi[rn + s], lo[rn + s]}, ps = {hi[rs + s], lo[rs + s]};
      const FF pe = {hi[r0 + se], lo[r0 + se]}, pw = {hi[r0 + sw], lo[r0 + sw]};
      const FF dn = (S[0] + S[3]) + (S[1] + S[2]), nn = n0f + dn;
      const FF mt = vb * (S[3] - S[0]) + va * (S[2] - S[1]), mp = vb * OB + va * OA;
      const FF u2 = (mt * mt + mp * mp) / (nn * nn);
      const FF om = diff(one, p0) * (one + p0), g1 = diff(pn, ps) * gtf, g2 = diff(pe, pw) * gp;
      const FF dens = A4 * (om * om) + k2 * (g1 * g1 + g2 * g2);
      const float pm = fmaxf(fmaxf(fabsf(p0.h), fmaxf(fabsf(pn.h), fabsf(ps.h))), fmaxf(fabsf(pe.h), fabsf(pw.h)));
      // the comparisons are false for NaN; products below 1e-23 lose bits of their low word, which matters where they
      // are the largest |u|^2 so far, or the density of Psi itself
      if (nn.h >= 1e-6f && nn.h <= 1e6f && big <= 1e6f && pm <= 1e4f && u2.h <= 1e6f && dens.h <= 1e12f &&
          (u2.h >= 1e-23f || best.h >= 1e-23f || (mt.h == 0.0f && mp.h == 0.0f)) &&
          (dens.h >= 1e-23f || ((A4.h == 0.0f || om.h == 0.0f) && (k2.h == 0.0f || (g1.h == 0.0f && g2.h == 0.0f))))) {
        m = m + dn;
        const FF sh = two_sum(ph.h, p0.h), sl = two_sum(ph.l, p0.l), st = two_sum(sh.l, sl.h);
        ph = quick_sum(sh.h, st.h);
        ph3 = __fadd_rn(ph3, __fadd_rn(sl.l, st.l));
        psi = psi + dens;
        ++count;
        if (exceeds(u2, best)) {
          best = u2;
          best_at = r0 + s;
        }
      } else {
        node_totals(state, stride, coefd, nt, ns, q, s, A, kappa, n0, gt, vd, acc);
      }
    }
    const double dA = coefd[C_DA * nt + q];
    acc[0] += (to_d(m) + n0 * count) * dA;
    acc[1] += (to_d(ph) + (double)ph3) * dA;
    acc[2] += to_d(psi) * dA;
  }
  // the CTA's node of the largest |u|^2 again in FP64, by one thread
  __shared__ FF s_best[TOTAL_THREADS / 32];
  __shared__ int64_t s_at[TOTAL_THREADS / 32];
  for (int o = 16; o > 0; o >>= 1) {
    const FF x = {__shfl_down_sync(0xffffffffu, best.h, o), __shfl_down_sync(0xffffffffu, best.l, o)};
    const int64_t at = __shfl_down_sync(0xffffffffu, best_at, o);
    if (exceeds(x, best)) {
      best = x;
      best_at = at;
    }
  }
  if ((threadIdx.x & 31) == 0) {
    s_best[threadIdx.x >> 5] = best;
    s_at[threadIdx.x >> 5] = best_at;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < TOTAL_THREADS / 32; ++w)
      if (exceeds(s_best[w], best)) {
        best = s_best[w];
        best_at = s_at[w];
      }
    if (best_at >= 0) {
      double nn, a, b;
      node_moments(state, stride, best_at, vd, n0, nn, a, b);
      acc[3] = fmax(acc[3], a * a + b * b);
    }
  }
  acc[3] = sqrt(acc[3]);
  reduce_totals(acc, partials);
}

// L_I: the interface edges of every row counted, then weighted in FP64 (r dtheta across varphi, the row's
// edge length across theta).  The sign of an FP32 phi is that of the float pair's high word, or of the sum where that
// word alone does not tell (0; an infinity, whose low word is NaN in a state that has diverged).
__device__ __forceinline__ bool crosses(double a, double b) { return a * b < 0.0; }
__device__ __forceinline__ bool crosses(float a, float b) { return (a < 0.0f && b > 0.0f) || (a > 0.0f && b < 0.0f); }
__device__ __forceinline__ double phi_sign(const double* state, int64_t stride, int64_t idx) {
  return state[NPOP * stride + idx];
}
__device__ __forceinline__ float phi_sign(const float* state, int64_t stride, int64_t idx) {
  const float h = state[NPOP * stride + idx];
  return h != 0.0f && isfinite(h) ? h : h + state[(NPOP + 1) * stride + idx];
}
template <typename T>
__global__ void __launch_bounds__(TOTAL_THREADS) interface_kernel(const T* state, int64_t stride, const double* coefd,
                                                                  int nt, int ns, int W, int segs, int len,
                                                                  double edge_p, double* partials) {
  const int c = threadIdx.x & (W - 1), rb = TOTAL_THREADS / W;
  double acc = 0.0;
  for (int64_t unit = blockIdx.x * (int64_t)rb + threadIdx.x / W; unit < (int64_t)nt * segs;
       unit += (int64_t)gridDim.x * rb) {
    const int q = (int)(unit / segs), first = (int)(unit - (int64_t)q * segs) * len;
    const int last = first + len < ns ? first + len : ns;
    const int64_t r0 = (int64_t)q * ns, rn = (int64_t)(q + 1 < nt ? q + 1 : 0) * ns;
    int np = 0, nn = 0;
    for (int s = first + c; s < last; s += W) {
      const T p0 = phi_sign(state, stride, r0 + s);
      np += crosses(p0, phi_sign(state, stride, r0 + (s + 1 < ns ? s + 1 : 0))) ? 1 : 0;
      nn += crosses(p0, phi_sign(state, stride, rn + s)) ? 1 : 0;
    }
    if (np | nn) acc += edge_p * np + coefd[C_EDGE * nt + q] * nn;
  }
  __shared__ double red[TOTAL_THREADS];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int w = TOTAL_THREADS / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) partials[blockIdx.x] = red[0];
}

// Fixed-order sum (or max) of part[b * stride + k] over b < nb by one warp: lane l takes b = l, l + 32,
// ... in order, then a shuffle tree; the result depends only on nb, not on scheduling.
__device__ __forceinline__ double warp_fold(const double* part, int nb, int stride, int k, bool is_max) {
  const int lane = threadIdx.x & 31;
  double x = 0.0;
  for (int b = lane; b < nb; b += 32) {
    const double v = part[b * stride + k];
    x = is_max ? fmax(x, v) : x + v;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double y = __shfl_down_sync(0xffffffffu, x, o);
    x = is_max ? fmax(x, y) : x + y;
  }
  return x;
}

__global__ void interface_final_kernel(const double* partials, int nb, double* out) {
  const double x = warp_fold(partials, nb, 1, 0, false);
  if (threadIdx.x == 0) *out = x;
}

// one warp per output k (blockDim = 32 NTOT)
__global__ void totals_final_kernel(const double* partials, int nb, double* out) {
  const int k = threadIdx.x >> 5;
  const double x = warp_fold(partials, nb, NSUM, k, k == 3);
  if ((threadIdx.x & 31) == 0) out[k] = x;
}

__device__ __forceinline__ float mul_rn(float x, float y) { return __fmul_rn(x, y); }
__device__ __forceinline__ double mul_rn(double x, double y) { return __dmul_rn(x, y); }

// The surrogate's snapshot kernels work in the state's own precision T (they run once per window).
template <typename T>
__device__ __forceinline__ void node_moments_t(const T* state, int64_t stride, int64_t idx, const VD& vd, T n0, T& n,
                                               T& ut, T& up) {
  T row[4] = {0, 0, 0, 0}, col[4] = {0, 0, 0, 0};
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const T x = state[(4 * i + j) * stride + idx];
      row[i] += x;
      col[j] += x;
    }
  n = n0 + ((row[0] + row[1]) + (row[2] + row[3]));
  ut = ((T)vd.v[0] * row[0] + (T)vd.v[1] * row[1] + (T)vd.v[2] * row[2] + (T)vd.v[3] * row[3]) / n;
  up = ((T)vd.v[0] * col[0] + (T)vd.v[1] * col[1] + (T)vd.v[2] * col[2] + (T)vd.v[3] * col[3]) / n;
}

// (phi, n, u_theta, u_phi) per node, from the state, as FP32.
template <typename T>
__global__ void snapshot_out_kernel(const T* state, int64_t stride, int64_t n, T n0, float* snap, VD vd) {
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n; idx += (int64_t)gridDim.x * blockDim.x) {
    T nn, a, b;
    node_moments_t(state, stride, idx, vd, n0, nn, a, b);
    reinterpret_cast<float4*>(snap)[idx] =
        make_float4((float)load_phi(state, stride, idx), (float)nn, (float)a, (float)b);
  }
}

// Per-block FP64 partial sums of n dA and phi dA over a snapshot (dA the row's area element).
__global__ void __launch_bounds__(TOTAL_THREADS) snapshot_sums_kernel(const float* snap, const double* coefd, int nt,
                                                                      int ns, double* partials) {
  const int64_t n = (int64_t)nt * ns;
  double sn = 0.0, sp = 0.0;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n; idx += (int64_t)gridDim.x * blockDim.x) {
    const float4 v = reinterpret_cast<const float4*>(snap)[idx];
    const double dA = coefd[C_DA * nt + (int)(idx / ns)];
    sn += (double)v.y * dA;
    sp += (double)v.x * dA;
  }
  for (int o = 16; o > 0; o >>= 1) {
    sn += __shfl_down_sync(0xffffffffu, sn, o);
    sp += __shfl_down_sync(0xffffffffu, sp, o);
  }
  __shared__ double red[2][TOTAL_THREADS / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    red[0][wid] = sn;
    red[1][wid] = sp;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double x = 0.0;
    for (int w = 0; w < TOTAL_THREADS / 32; ++w) x += red[threadIdx.x][w];
    partials[blockIdx.x * NSUM + threadIdx.x] = x;
  }
}

// shift[0] = (mass - sum n dA) / area, shift[1] = (phi_total - sum phi dA) / area (Sec. 2.5 totals);
// one warp per total (blockDim = 64).
__global__ void snapshot_shift_kernel(const double* partials, int nb, double mass, double phi_total, double inv_area,
                                      double* shift) {
  const int k = threadIdx.x >> 5;
  const double x = warp_fold(partials, nb, NSUM, k, false);
  if ((threadIdx.x & 31) == 0) shift[k] = ((k == 0 ? mass : phi_total) - x) * inv_area;
}

// The surrogate restart from a snapshot (n', u', phi'), with n' += shift[0] and phi' += shift[1] when
// shift != NULL.  keep_neq == 0: f := f^eq(n', u') (Eq. feq).  keep_neq != 0: f := f + f^eq(n', u') -
// f^eq(n, u) with (n, u) the moments of the current f, which keeps the non-equilibrium part f - f^eq
// of the state and gives f the moments (n', u').  In the deviation storage g = f - n0 w_i w_j:
// f^eq - n0 w_i w_j = w_i w_j ((n - n0) + n P(u)), P(u) = xi + (xi^2 - u^2)/2 + xi (xi^2 - 3 u^2)/6.
template <typename T>
__global__ void snapshot_in_kernel(T* state, int64_t stride, int64_t n, T n0, const float* snap, const double* shift,
                                   int keep_neq, VD vd) {
  const T dn = shift ? (T)shift[0] : (T)0, dphi = shift ? (T)shift[1] : (T)0;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n; idx += (int64_t)gridDim.x * blockDim.x) {
    const float4 s = reinterpret_cast<const float4*>(snap)[idx];
    const T nn = (T)s.y + dn, a = (T)s.z, b = (T)s.w;
    const T usq = a * a + b * b;
    T n1 = 0, a1 = 0, b1 = 0, usq1 = 0;
    if (keep_neq) {
      node_moments_t(state, stride, idx, vd, n0, n1, a1, b1);
      usq1 = a1 * a1 + b1 * b1;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const T vi = (T)vd.v[i], vj = (T)vd.v[j], ww = (T)(vd.w[i] * vd.w[j]);
        const T xi = vi * a + vj * b;
        const T pm = xi + (T)0.5 * (xi * xi - usq) + xi * (xi * xi - (T)3 * usq) / (T)6;
        T* g = state + (4 * i + j) * stride + idx;
        if (keep_neq) {
          const T xi1 = vi * a1 + vj * b1;
          const T pm1 = xi1 + (T)0.5 * (xi1 * xi1 - usq1) + xi1 * (xi1 * xi1 - (T)3 * usq1) / (T)6;
          // rounded products (no contraction): the state's own moments give exactly zero change
          *g = *g + ww * ((nn - n1) + (mul_rn(nn, pm) - mul_rn(n1, pm1)));
        } else {
          *g = ww * ((nn - n0) + nn * pm);
        }
      }
    store_phi(state, stride, idx, (double)s.x + (double)dphi);
  }
}

int grid_for(int64_t n) {
  int64_t g = (n + 255) / 256;
  if (g > 152 * 16) g = 152 * 16;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

int totals_blocks() { return TOTAL_BLOCKS; }

__device__ const RowRules<double> g_pair_rules = make_row_rules<double>();

// One entry a thread: a host loop over them took 65 us of vlb_create at 1024 rows and 235 us at 4096.
__global__ void __launch_bounds__(128) pair_rows_kernel(const double* coefd, int nt, double dt, double M, double kappa,
                                                        float* rows) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= nt * kRowTable) return;  // whole warps: a row each
  const int q = x / kRowTable;
  const RowRule<double> r = g_pair_rules.e[x % kRowTable];
  const double s = r.s == 3 ? 1.0 : r.s == 2 ? kappa : (r.s == 1 ? dt * M : dt);
  const double y = r.y ? coefd[C_J * nt + (q + r.y - 3 + nt) % nt] : 1.0;
  rows[x] = row_table_entry(s * (r.c1 * coefd[r.x1 * nt + q] * y + r.c2 * coefd[r.x2 * nt + q]), x % kRowTable);
}

cudaError_t launch_pair_rows(const double* coefd, int nt, double dt, double M, double kappa, float* rows,
                             cudaStream_t s) {
  pair_rows_kernel<<<(nt * kRowTable + 127) / 128, 128, 0, s>>>(coefd, nt, dt, M, kappa, rows);
  return cudaGetLastError();
}

// out[q] = sum over s of x[q][s], one CTA per row: each thread adds its strided elements in order,
// then a fixed-order tree in shared memory (deterministic).
__global__ void __launch_bounds__(256) row_sums_kernel(const double* x, int ns, double* out) {
  __shared__ double red[256];
  const double* row = x + (int64_t)blockIdx.x * ns;
  double acc = 0.0;
  for (int s = threadIdx.x; s < ns; s += blockDim.x) acc += row[s];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = red[0];
}

cudaError_t launch_row_sums(const double* x, int nt, int ns, double* out, cudaStream_t s) {
  row_sums_kernel<<<nt, 256, 0, s>>>(x, ns, out);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_init_feq(T* state, int64_t stride, const double* rho, const double* ut, const double* up,
                            const double* phi, int64_t n, double n0, cudaStream_t s) {
  init_feq_kernel<T><<<grid_for(n), 256, 0, s>>>(state, stride, rho, ut, up, phi, n, n0, make_vd());
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_convert_in(T* state, int64_t stride, const double* src, int64_t n, double n0, cudaStream_t s) {
  convert_in_kernel<T><<<grid_for(n * NARR), 256, 0, s>>>(state, stride, src, n, n0, make_vd());
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_convert_out(double* dst, const T* state, int64_t stride, int64_t n, double n0, cudaStream_t s) {
  convert_out_kernel<T><<<grid_for(n * NARR), 256, 0, s>>>(dst, state, stride, n, n0, make_vd());
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_fields(const T* state, int64_t stride, const double* coefd, int nt, int ns, double A, double kappa,
                          double n0, double* rho, double* ut, double* up, double* phi, double* mu, cudaStream_t s) {
  fields_kernel<T><<<dim3((ns + 255) / 256, nt), 256, 0, s>>>(state, stride, coefd, nt, ns, A, kappa, n0, rho, ut, up,
                                                             phi, mu, make_vd());
  return cudaGetLastError();
}

// How the sums over rows are shared out: W threads (a power of two up to a CTA) to a segment, and rows cut into
// segments of whole passes of W nodes where they alone would leave CTAs idle (few long rows: 8 x 262144 is 8 CTAs
// of 1024 passes otherwise).
struct RowSplit {
  int W, segs, len, blocks;
};
static RowSplit row_split(int nt, int ns, int n_blocks) {
  RowSplit r;
  r.W = 1;
  while (r.W < TOTAL_THREADS && r.W < ns) r.W *= 2;
  const int rb = TOTAL_THREADS / r.W;
  const int64_t units = (int64_t)n_blocks * rb, passes = (ns + r.W - 1) / r.W;
  const int64_t want = units / nt > 1 ? (units / nt < passes ? units / nt : passes) : 1;
  const int64_t per = (passes + want - 1) / want;
  r.len = (int)(per * r.W);
  r.segs = (int)((passes + per - 1) / per);
  const int64_t blocks = ((int64_t)nt * r.segs + rb - 1) / rb;
  r.blocks = (int)(blocks < n_blocks ? blocks : n_blocks);
  return r;
}

template <typename T>
cudaError_t launch_totals(const T* state, int64_t stride, const double* coefd, int nt, int ns, double r, double A,
                          double kappa, double n0, double* partials, int n_blocks, double* out, cudaStream_t s) {
  const double gt = 1.0 / (2.0 * r * (2.0 * M_PI / nt));
  if constexpr (sizeof(T) == 4) {
    const RowSplit r = row_split(nt, ns, n_blocks);
    n_blocks = r.blocks;
    totals32_kernel<<<n_blocks, TOTAL_THREADS, 0, s>>>(state, stride, coefd, nt, ns, r.W, r.segs, r.len, A, kappa, n0,
                                                       gt, partials, make_vd());
  } else {
    totals_kernel<T><<<n_blocks, TOTAL_THREADS, 0, s>>>(state, stride, coefd, nt, ns, A, kappa, n0, gt, partials,
                                                        make_vd());
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  totals_final_kernel<<<1, 32 * NTOT, 0, s>>>(partials, n_blocks, out);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_interface(const T* state, int64_t stride, const double* coefd, int nt, int ns, double r,
                             double* partials, int n_blocks, double* out, cudaStream_t s) {
  const RowSplit w = row_split(nt, ns, n_blocks);
  n_blocks = w.blocks;
  interface_kernel<T><<<n_blocks, TOTAL_THREADS, 0, s>>>(state, stride, coefd, nt, ns, w.W, w.segs, w.len,
                                                         r * (2.0 * M_PI / nt), partials);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  interface_final_kernel<<<1, 32, 0, s>>>(partials, n_blocks, out);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_snapshot_out(const T* state, int64_t stride, int64_t n, double n0, float* snap, cudaStream_t s) {
  snapshot_out_kernel<T><<<grid_for(n), 256, 0, s>>>(state, stride, n, (T)n0, snap, make_vd());
  return cudaGetLastError();
}

cudaError_t launch_snapshot_shift(const float* snap, const double* coefd, int nt, int ns, double mass,
                                  double phi_total, double inv_area, double* partials, double* shift, cudaStream_t s) {
  snapshot_sums_kernel<<<TOTAL_BLOCKS, TOTAL_THREADS, 0, s>>>(snap, coefd, nt, ns, partials);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  snapshot_shift_kernel<<<1, 64, 0, s>>>(partials, TOTAL_BLOCKS, mass, phi_total, inv_area, shift);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_snapshot_in(T* state, int64_t stride, int64_t n, double n0, const float* snap, const double* shift,
                               int keep_neq, cudaStream_t s) {
  snapshot_in_kernel<T><<<grid_for(n), 256, 0, s>>>(state, stride, n, (T)n0, snap, shift, keep_neq, make_vd());
  return cudaGetLastError();
}

#define VLB_INST(T)                                                                                              \
  template cudaError_t launch_init_feq<T>(T*, int64_t, const double*, const double*, const double*,              \
                                          const double*, int64_t, double, cudaStream_t);                          \
  template cudaError_t launch_convert_in<T>(T*, int64_t, const double*, int64_t, double, cudaStream_t);         \
  template cudaError_t launch_convert_out<T>(double*, const T*, int64_t, int64_t, double, cudaStream_t);        \
  template cudaError_t launch_fields<T>(const T*, int64_t, const double*, int, int, double, double, double,     \
                                        double*, double*, double*, double*, double*, cudaStream_t);               \
  template cudaError_t launch_totals<T>(const T*, int64_t, const double*, int, int, double, double, double,      \
                                        double, double*, int, double*, cudaStream_t);                            \
  template cudaError_t launch_interface<T>(const T*, int64_t, const double*, int, int, double, double*, int,     \
                                           double*, cudaStream_t);                                                \
  template cudaError_t launch_snapshot_out<T>(const T*, int64_t, int64_t, double, float*, cudaStream_t);        \
  template cudaError_t launch_snapshot_in<T>(T*, int64_t, int64_t, double, const float*, const double*, int,   \
                                             cudaStream_t);
VLB_INST(float)
VLB_INST(double)
#undef VLB_INST

}  // namespace vlb
