// Stabilised semi-implicit Cahn-Hilliard stage (not part of the paper's method, which advances Eq. CH
// explicitly; the explicit step is limited to dt ~ h^4 / (M kappa)).
//
// With the stabilisation the phi part of every SSP-RK3 stage reads
//   phi_out = phi^n + b (phi_in - phi^n + P(dt L_phi(phi_in))),   (first stage: phi^n = phi_in, b = 1)
// with the fixed preconditioner P = J^{-1} (I + dt M kappa D^2)^{-1} J, D the constant-coefficient
// periodic five-point Laplacian at the finest spacings of the grid (h_theta = r dtheta, h_phi =
// (R - r) dvarphi on the torus, R dvarphi flat).  P is diagonal in the discrete Fourier basis of J x:
// a mode (m, n) is divided by 1 + dt M kappa lambda(m, n) with lambda = ((4/h_theta^2) sin^2(pi m/N_theta)
// + (4/h_phi^2) sin^2(pi n/N_phi))^2; the mean (m = n = 0) is kept, so P conserves sum J x (the
// integral of x sqrt(g)).  The stage kernel writes dt L_phi into a scratch array; three kernels then
//   1. transform the theta rows of J dt L_phi, two rows as one complex transform per CTA, and store the
//      half spectrum n = 0 .. N_phi / 2 (the two real columns 0 and N_phi / 2 packed into one),
//   2. transform strips of columns, divide by 1 + dt M kappa lambda and transform them back,
//   3. transform the rows back (FP64: two at a time), divide by N_theta N_phi J and form phi_out (in FP32 as
//      the float pair hi + lo with an error-free sum, as the stage kernel does).
// The FFTs are in place in shared memory, in the state's precision; N_theta and N_phi are powers of
// two <= 4096.  The two factors of lambda, (4/h_theta^2) sin^2(pi m/N_theta) and (4/h_phi^2)
// sin^2(pi n/N_phi), are tabulated once in FP64 on the host (ch_stab_tables) and rounded to the state
// precision, so the division runs in that precision with no transcendental per mode; so are the twiddles of both
// transform lengths, which each CTA copies from global memory (L2) into shared memory.
// The kernels are bound by the shared-memory passes and the barriers of the transforms, so half the data is
// half the time: per stage at 1024 x 2048 in FP32 20.5 + 41.7 + 26.9 us with complex transforms of every row,
// 13.6 + 21.2 + 24.1 us now.
#include <math.h>

#include <vector>

#include "vlb_internal.cuh"

namespace vlb {

namespace {

template <typename T>
struct C2 {
  T x, y;
};

__device__ __forceinline__ int bitrev(int i, int logn) { return (int)(__brev((unsigned)i) >> (32 - logn)); }

// Twiddles stored level by level, so that the butterflies of one level read consecutive entries
// (a single table indexed by j n / 2^l puts a warp's reads on one shared-memory bank at the middle
// levels): tw[2^(l-1) - 1 + j] = exp(-2 pi i j / 2^l), j < 2^(l-1), l = 1 .. log2 n; n - 1 entries.

// Shared-memory position of element e of a row transform: one pad element every 2^sh elements, so
// that the bit-reversed scatter of 32 consecutive indices (multiples of n / 32) and the butterflies
// spread over the banks.  Column strips use sh = 31 (no padding).
__device__ __forceinline__ int padded(int e, int sh) { return e + (e >> sh); }
__host__ __device__ inline int row_pad_shift(int logn) { return logn >= 5 ? logn - 5 : 31; }

template <typename T>
__device__ __forceinline__ C2<T> cmul(C2<T> v, C2<T> t) {
  return {v.x * t.x - v.y * t.y, v.x * t.y + v.y * t.x};
}
// c + a b
template <typename T>
__device__ __forceinline__ C2<T> cfma(C2<T> a, C2<T> b, C2<T> c) {
  return {fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y))};
}

// In-place FFT along the first index of a[i * w + c] (w = 2^logw interleaved sequences of length n,
// loaded in bit-reversed order of i; element e stored at padded(e, sh)), decimation in time: the
// radix-2 levels l = 1 .. log2 n, taken two at a time as one radix-4 pass (one radix-2 pass first when
// log2 n is odd), which halves the shared-memory passes and barriers.  A radix-4 group of levels
// (l, l + 1) holds the elements i0 + {0, 1, 2, 3} h (h = 2^(l-1), i0 = 4h (g / h) + g % h, j = g % h):
// level l pairs (0, 1) and (2, 3) with twiddle t1 = W_2h^j, level l + 1 pairs (0, 2) with
// t2 = W_4h^j and (1, 3) with W_4h^(j + h) = -i t2 (+i t2 for the inverse).  inverse: conjugate
// twiddles (unnormalised).
template <typename T>
__device__ void fft_strided(C2<T>* a, int n, int logn, int logw, int sh, const C2<T>* tw, bool inverse) {
  const int w = 1 << logw;
  int l = 1;
  if (logn & 1) {  // level 1 alone: pairs (2 g, 2 g + 1), twiddle 1
    const int nb = (n >> 1) << logw;
    for (int idx = threadIdx.x; idx < nb; idx += blockDim.x) {
      const int g = idx >> logw, c = idx & (w - 1);
      const int e0 = padded(((2 * g) << logw) + c, sh), e1 = padded(((2 * g + 1) << logw) + c, sh);
      const C2<T> u = a[e0], v = a[e1];
      a[e0] = {u.x + v.x, u.y + v.y};
      a[e1] = {u.x - v.x, u.y - v.y};
    }
    __syncthreads();
    l = 2;
  }
  const int nq = (n >> 2) << logw;
  for (; l < logn; l += 2) {
    const int h = 1 << (l - 1);
    for (int idx = threadIdx.x; idx < nq; idx += blockDim.x) {
      const int g = idx >> logw, c = idx & (w - 1);
      const int j = g & (h - 1);
      const int i0 = ((g >> (l - 1)) << (l + 1)) + j;
      C2<T> t1 = tw[h - 1 + j], t2 = tw[2 * h - 1 + j];
      if (inverse) {
        t1.y = -t1.y;
        t2.y = -t2.y;
      }
      const int e0 = padded((i0 << logw) + c, sh), e1 = padded(((i0 + h) << logw) + c, sh);
      const int e2 = padded(((i0 + 2 * h) << logw) + c, sh), e3 = padded(((i0 + 3 * h) << logw) + c, sh);
      // multiply-adds throughout: as many operations as products and sums apart, two roundings instead of three
      const C2<T> a0 = a[e0], a1 = a[e1], a2 = a[e2], a3 = a[e3];
      const C2<T> n1 = {-t1.x, -t1.y}, b0 = cfma(a1, t1, a0), b1 = cfma(a1, n1, a0);
      const C2<T> b2 = cfma(a3, t1, a2), b3 = cfma(a3, n1, a2);
      const C2<T> t3 = inverse ? C2<T>{-t2.y, t2.x} : C2<T>{t2.y, -t2.x};  // +i t2 / -i t2
      a[e0] = cfma(b2, t2, b0);
      a[e2] = cfma(b2, C2<T>{-t2.x, -t2.y}, b0);
      a[e1] = cfma(b3, t3, b1);
      a[e3] = cfma(b3, C2<T>{-t3.x, -t3.y}, b1);
    }
    __syncthreads();
  }
}

// The adjoint of fft_strided (the unnormalised inverse transform) with the passes in reverse: natural order in,
// bit-reversed order out (element e ends at position bitrev(e)), so that a transform and its inverse need no
// reordering in between.
template <typename T>
__device__ void fft_adjoint(C2<T>* a, int n, int logn, int logw, int sh, const C2<T>* tw) {
  const int w = 1 << logw, nq = (n >> 2) << logw;
  for (int l = logn - 1; l >= 1 + (logn & 1); l -= 2) {
    const int h = 1 << (l - 1);
    for (int idx = threadIdx.x; idx < nq; idx += blockDim.x) {
      const int g = idx >> logw, c = idx & (w - 1);
      const int j = g & (h - 1);
      const int i0 = ((g >> (l - 1)) << (l + 1)) + j;
      const C2<T> t1 = {tw[h - 1 + j].x, -tw[h - 1 + j].y}, t2 = {tw[2 * h - 1 + j].x, -tw[2 * h - 1 + j].y};
      const int e0 = padded((i0 << logw) + c, sh), e1 = padded(((i0 + h) << logw) + c, sh);
      const int e2 = padded(((i0 + 2 * h) << logw) + c, sh), e3 = padded(((i0 + 3 * h) << logw) + c, sh);
      const C2<T> y0 = a[e0], y1 = a[e1], y2 = a[e2], y3 = a[e3];
      const C2<T> b0 = {y0.x + y2.x, y0.y + y2.y}, b1 = {y1.x + y3.x, y1.y + y3.y};
      const C2<T> c2 = cmul(C2<T>{y0.x - y2.x, y0.y - y2.y}, t2);
      C2<T> c3 = cmul(C2<T>{y1.x - y3.x, y1.y - y3.y}, t2);
      c3 = {-c3.y, c3.x};  // times +i
      a[e0] = {b0.x + b1.x, b0.y + b1.y};
      a[e1] = cmul(C2<T>{b0.x - b1.x, b0.y - b1.y}, t1);
      a[e2] = {c2.x + c3.x, c2.y + c3.y};
      a[e3] = cmul(C2<T>{c2.x - c3.x, c2.y - c3.y}, t1);
    }
    __syncthreads();
  }
  if (logn & 1) {
    const int nb = (n >> 1) << logw;
    for (int idx = threadIdx.x; idx < nb; idx += blockDim.x) {
      const int g = idx >> logw, c = idx & (w - 1);
      const int e0 = padded(((2 * g) << logw) + c, sh), e1 = padded(((2 * g + 1) << logw) + c, sh);
      const C2<T> u = a[e0], v = a[e1];
      a[e0] = {u.x + v.x, u.y + v.y};
      a[e1] = {u.x - v.x, u.y - v.y};
    }
    __syncthreads();
  }
}

constexpr int kBatch = 8;  // global loads a thread keeps in flight before it stores them

// the n - 1 per-level twiddles of a transform, from the host-computed table
template <typename T>
__device__ __forceinline__ void load_twiddles(C2<T>* tw, const C2<T>* table, int n) {
  for (int k0 = threadIdx.x; k0 < n - 1; k0 += kBatch * blockDim.x) {
    C2<T> v[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int k = k0 + u * blockDim.x;
      if (k < n - 1) v[u] = table[k];
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int k = k0 + u * blockDim.x;
      if (k < n - 1) tw[k] = v[u];
    }
  }
}

// 1. Rows q = 2 b and q + 1 of J dt L_phi, packed as the real and imaginary part of one transform, -> their
// spectra at 0 .. N_phi / 2 - 1 (the others are their conjugates), entry 0 holding the real values at 0 and N_phi / 2.
template <typename T>
__global__ void __launch_bounds__(256) row_fwd_kernel(int ns, int logns, const T* dphi, const double* J,
                                                      const C2<T>* tw_s, C2<T>* buf) {
  extern __shared__ __align__(16) unsigned char raw[];
  C2<T>* a = reinterpret_cast<C2<T>*>(raw);
  const int sh = row_pad_shift(logns), nh = ns / 2;
  C2<T>* tw = a + padded(ns, sh);
  const int64_t q = 2 * (int64_t)blockIdx.x;
  const T j0 = (T)J[q], j1 = (T)J[q + 1];
  const T *x0 = dphi + q * ns, *x1 = x0 + ns;
  for (int s0 = threadIdx.x; s0 < ns; s0 += (kBatch / 2) * blockDim.x) {
    T v[kBatch / 2], w[kBatch / 2];
#pragma unroll
    for (int u = 0; u < kBatch / 2; ++u) {
      const int s = s0 + u * blockDim.x;
      if (s < ns) {
        v[u] = x0[s];
        w[u] = x1[s];
      }
    }
#pragma unroll
    for (int u = 0; u < kBatch / 2; ++u) {
      const int s = s0 + u * blockDim.x;
      if (s < ns) a[padded(bitrev(s, logns), sh)] = {j0 * v[u], j1 * w[u]};
    }
  }
  load_twiddles(tw, tw_s, ns);
  __syncthreads();
  fft_strided(a, ns, logns, 0, sh, tw, false);
  C2<T>*r0 = buf + q * nh, *r1 = r0 + nh;
  for (int k = threadIdx.x; k < nh; k += blockDim.x) {
    const C2<T> z = a[padded(k, sh)], y = a[padded(k ? ns - k : nh, sh)];
    if (k == 0) {
      r0[0] = {z.x, y.x};
      r1[0] = {z.y, y.y};
    } else {  // (z + conj y) / 2 and (z - conj y) / 2i
      r0[k] = {T(0.5) * (z.x + y.x), T(0.5) * (z.y - y.y)};
      r1[k] = {T(0.5) * (z.y + y.y), T(0.5) * (y.x - z.x)};
    }
  }
}

// 2. Columns n0 .. n0 + cw - 1 of the half spectrum: F_theta, division by 1 + s lambda(m, n), inverse F_theta.
template <typename T>
__global__ void __launch_bounds__(512) col_solve_kernel(int nt, int lognt, int nh, int lcw, T sfac, const T* lam_t,
                                                        const T* lam_p, const C2<T>* tw_t, C2<T>* buf) {
  extern __shared__ __align__(16) unsigned char raw[];
  C2<T>* a = reinterpret_cast<C2<T>*>(raw);
  const int cw = 1 << lcw;
  C2<T>* tw = a + ((size_t)nt << lcw);
  const int n0 = blockIdx.x << lcw;
  const int total = nt << lcw;
  for (int i0 = threadIdx.x; i0 < total; i0 += kBatch * blockDim.x) {
    C2<T> v[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int idx = i0 + u * blockDim.x;
      if (idx < total) v[u] = buf[(int64_t)(idx >> lcw) * nh + n0 + (idx & (cw - 1))];
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int idx = i0 + u * blockDim.x;
      if (idx < total) a[(bitrev(idx >> lcw, lognt) << lcw) + (idx & (cw - 1))] = v[u];
    }
  }
  load_twiddles(tw, tw_t, nt);
  __syncthreads();
  fft_strided(a, nt, lognt, lcw, 31, tw, false);
  auto damp = [&](int m, T lp) {
    const T lap = lam_t[m] + lp;
    return T(1) / (T(1) + sfac * lap * lap);
  };
  const int n = n0 + (threadIdx.x & (cw - 1));  // a thread keeps its column (blockDim % cw == 0)
  const T lp = lam_p[n];
  if (n) {
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
      const T g = damp(idx >> lcw, lp);
      a[idx].x *= g;
      a[idx].y *= g;
    }
  } else {
    // the real columns 0 and N_phi / 2 packed as c = f + i h: g_0 f + i g_h h = (g_0 + g_h) / 2 c(m) +
    // (g_0 - g_h) / 2 conj c(-m); the modes m and -m (the same damping) together
    const T lh = lam_p[nh];
    for (int idx = threadIdx.x; idx < (nt / 2 + 1) << lcw; idx += blockDim.x) {
      const int m = idx >> lcw, mr = m ? nt - m : 0;
      const T g0 = damp(m, lp), gh = damp(m, lh), p = T(0.5) * (g0 + gh), d = T(0.5) * (g0 - gh);
      const C2<T> z = a[m << lcw], y = a[mr << lcw];
      a[m << lcw] = {p * z.x + d * y.x, p * z.y - d * y.y};
      if (mr != m) a[mr << lcw] = {p * y.x + d * z.x, p * y.y - d * z.y};
    }
  }
  __syncthreads();
  fft_adjoint(a, nt, lognt, lcw, 31, tw);
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int q = idx >> lcw, c = idx & (cw - 1);
    buf[(int64_t)q * nh + n0 + c] = a[(bitrev(q, lognt) << lcw) + c];
  }
}

// (hi, lo) <- (base, base_lo) + inc with an error-free sum, renormalised (FP32 float pair)
__device__ __forceinline__ void pair_add(float base, float base_lo, float inc, float& hi, float& lo) {
  const float s1 = base + inc;
  const float bb = s1 - base;
  const float err = (base - (s1 - bb)) + (inc - bb);
  const float lo2 = base_lo + err;
  hi = s1 + lo2;
  lo = lo2 - (hi - s1);
}

// Rows that share an inverse transform.  In FP64 two, as real and imaginary part.  In FP32 one: the rounding of this
// transform is what phi keeps undamped, and with a row alone half of it goes with the imaginary part (populations at
// 1024 x 2048 after two steps: error 2.2e-7 with two rows, 1.9e-7 with one).
template <typename T>
constexpr int inv_rows() { return sizeof(T) == 8 ? 2 : 1; }

// 3. Rows q .. q + inv_rows - 1: inverse F_phi in one transform, y = Re (Im) / (N J), phi_out = phi^n + b (phi_in - phi^n + y).
template <typename T>
__global__ void __launch_bounds__(256) row_inv_kernel(int ns, int logns, double inv_n, const double* J,
                                                      const C2<T>* tw_s, const C2<T>* buf, const T* phin,
                                                      const T* phi0, T* phiout, int64_t lo_off, T b) {
  constexpr bool DF = sizeof(T) == 4;  // phi as a float pair
  constexpr int U = 4;                 // nodes per batch of loads (four state words each)
  constexpr int ROWS = inv_rows<T>(), NB = kBatch / ROWS;
  extern __shared__ __align__(16) unsigned char raw[];
  C2<T>* a = reinterpret_cast<C2<T>*>(raw);
  const int sh = row_pad_shift(logns), nh = ns / 2;
  C2<T>* tw = a + padded(ns, sh);
  const int64_t q = ROWS * (int64_t)blockIdx.x;
  const C2<T>*r0 = buf + q * nh, *r1 = r0 + nh;
  for (int s0 = threadIdx.x; s0 < nh; s0 += NB * blockDim.x) {
    C2<T> v[NB], w[NB];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int s = s0 + u * blockDim.x;
      if (s < nh) {
        v[u] = r0[s];
        w[u] = ROWS == 2 ? r1[s] : C2<T>{T(0), T(0)};
      }
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int s = s0 + u * blockDim.x;
      if (s >= nh) continue;
      if (s == 0) {  // the packed real values at 0 and N_phi / 2
        a[0] = {v[u].x, w[u].x};
        a[padded(bitrev(nh, logns), sh)] = {v[u].y, w[u].y};
      } else {  // x + i y and, at -s, conj x + i conj y
        a[padded(bitrev(s, logns), sh)] = {v[u].x - w[u].y, v[u].y + w[u].x};
        a[padded(bitrev(ns - s, logns), sh)] = {v[u].x + w[u].y, w[u].x - v[u].y};
      }
    }
  }
  load_twiddles(tw, tw_s, ns);
  __syncthreads();
  fft_strided(a, ns, logns, 0, sh, tw, true);
  const T scale[2] = {(T)(inv_n / J[q]), (T)(inv_n / J[q + ROWS - 1])};
  for (int s0 = threadIdx.x; s0 < ROWS * ns; s0 += U * blockDim.x) {  // two rows follow each other
    T ph[U], lo[U], base[U], base_lo[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int s = s0 + u * blockDim.x;
      if (s < ROWS * ns) {
        const int64_t g = q * ns + s;
        ph[u] = phin[g];
        lo[u] = DF ? phin[g + lo_off] : T(0);
        base[u] = phi0 ? phi0[g] : ph[u];
        base_lo[u] = phi0 ? (DF ? phi0[g + lo_off] : T(0)) : lo[u];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int s = s0 + u * blockDim.x;
      if (s >= ROWS * ns) continue;
      const int64_t g = q * ns + s;
      const C2<T> z = a[padded(s & (ns - 1), sh)];
      const T y = ROWS == 1 || s < ns ? z.x * scale[0] : z.y * scale[1];
      const T inc = phi0 ? b * (((ph[u] - base[u]) + (lo[u] - base_lo[u])) + y) : y;
      if constexpr (DF) {
        float hi_o, lo_o;
        pair_add(base[u], base_lo[u], inc, hi_o, lo_o);
        phiout[g] = hi_o;
        phiout[g + lo_off] = lo_o;
      } else {
        phiout[g] = base[u] + inc;
      }
    }
  }
}

int ilog2(int n) {
  int l = 0;
  while ((1 << l) < n) ++l;
  return l;
}

template <typename K>
cudaError_t smem_attr(K kernel, size_t bytes, int& mask) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 32 && (mask & (1 << dev))) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess && dev < 32) mask |= 1 << dev;
  return e;
}

constexpr size_t kColBudget = 96 * 1024;  // shared bytes of a column strip (without twiddles)

}  // namespace

bool ch_stab_shape_ok(int nt, int ns) {
  auto pow2 = [](int n) { return n >= 4 && n <= 4096 && (n & (n - 1)) == 0; };
  return pow2(nt) && pow2(ns);
}

// the complex spectrum, then the tables: the two factors of lambda (N_theta + N_phi values) and the
// per-level twiddles of both transform lengths ((N_theta - 1) + (N_phi - 1) complex values)
size_t ch_stab_table_elems(int nt, int ns) { return (size_t)(nt + ns) + 2 * (size_t)(nt - 1 + ns - 1); }
size_t ch_stab_buffer_bytes(int nt, int ns, size_t esize) {
  return ((size_t)nt * ns * 2 + ch_stab_table_elems(nt, ns)) * esize;
}
size_t ch_stab_table_offset(int nt, int ns, size_t esize) { return (size_t)nt * ns * 2 * esize; }

void ch_stab_tables(int nt, int ns, double h_t, double h_p, size_t esize, void* host_out) {
  std::vector<double> v;
  v.reserve(ch_stab_table_elems(nt, ns));
  for (int i = 0; i < nt + ns; ++i) {
    const bool th = i < nt;
    const double sn = sin(M_PI * (th ? i : i - nt) / (th ? nt : ns));
    v.push_back((th ? 4.0 / (h_t * h_t) : 4.0 / (h_p * h_p)) * sn * sn);
  }
  // twiddles level by level: entry 2^(l-1) - 1 + j = exp(-2 pi i j / 2^l), j < 2^(l-1)
  for (int n : {nt, ns})
    for (int half = 1; half < n; half *= 2)
      for (int j = 0; j < half; ++j) {
        v.push_back(cos(M_PI * j / half));
        v.push_back(-sin(M_PI * j / half));
      }
  for (size_t i = 0; i < v.size(); ++i) {
    if (esize == 8)
      ((double*)host_out)[i] = v[i];
    else
      ((float*)host_out)[i] = (float)v[i];
  }
}

template <typename T>
cudaError_t launch_ch_stab(int nt, int ns, double dt_m_kappa, const double* J, const T* dphi, void* buf, const T* phin,
                           const T* phi0, T* phiout, int64_t lo_off, T b, cudaStream_t st) {
  if (!ch_stab_shape_ok(nt, ns)) return cudaErrorInvalidValue;
  const int lognt = ilog2(nt), logns = ilog2(ns);
  C2<T>* cb = reinterpret_cast<C2<T>*>(buf);
  const T* lam = reinterpret_cast<const T*>(buf) + (size_t)nt * ns * 2;  // ch_stab_tables
  const C2<T>* tw_t = reinterpret_cast<const C2<T>*>(lam + nt + ns);      // 8- or 16-byte aligned
  const C2<T>* tw_s = tw_t + (nt - 1);
  const size_t row_bytes = sizeof(C2<T>) * ((size_t)ns * 2 + 32);  // data (with its pads) and twiddles
  // column strips of 2^lcw columns: wide enough for whole 32-byte segments, narrow enough that the
  // launch keeps at least 256 CTAs of 512 threads (about two per SM) when the grid allows
  const int nh = ns / 2;
  int lcw = 0;
  while (lcw < 5 && (2 << lcw) <= nh && ((size_t)nt << lcw) * 2 * sizeof(C2<T>) <= kColBudget &&
         (lcw < 2 || (nh >> (lcw + 1)) >= 256))
    ++lcw;
  const size_t col_bytes = sizeof(C2<T>) * (((size_t)nt << lcw) + nt);
  const int col_threads = ((size_t)nt << lcw) >= 2048 ? 512 : 256;
  // the attribute is set once per device to the largest size any grid needs (setting it to a
  // smaller size would cap later launches on larger grids)
  constexpr size_t row_max = sizeof(C2<T>) * (4096 * 2 + 32);
  constexpr size_t col_max = kColBudget + sizeof(C2<T>) * 4096;
  static int m1 = 0, m2 = 0, m3 = 0;
  cudaError_t e;
  if ((e = smem_attr(row_fwd_kernel<T>, row_max, m1)) != cudaSuccess) return e;
  if ((e = smem_attr(col_solve_kernel<T>, col_max, m2)) != cudaSuccess) return e;
  if ((e = smem_attr(row_inv_kernel<T>, row_max, m3)) != cudaSuccess) return e;
  row_fwd_kernel<T><<<nt / 2, 256, row_bytes, st>>>(ns, logns, dphi, J, tw_s, cb);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  col_solve_kernel<T><<<nh >> lcw, col_threads, col_bytes, st>>>(nt, lognt, nh, lcw, (T)dt_m_kappa, lam, lam + nt, tw_t,
                                                                 cb);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  row_inv_kernel<T><<<nt / inv_rows<T>(), 256, row_bytes, st>>>(ns, logns, 1.0 / ((double)nt * ns), J, tw_s, cb, phin, phi0, phiout,
                                                   lo_off, b);
  return cudaGetLastError();
}

namespace {

// ---- Structure factor S(m, n) = |F phi|^2 and its two sums (the L_S diagnostic) --------------------
// The same transforms in FP64 whatever the state's precision (phi in FP32 is the float pair hi + lo, exact in a
// double).  Bound by the FP64 units, so phi's realness is used throughout: two rows share one complex
// transform, only the columns n = 0 .. N_phi / 2 are kept (columns 0 and N_phi / 2, real per row, packed
// into one), the mirrored half enters by weight 2, and one root serves the modes m and -m.  A column CTA sums
// S and |k| S over its strip (k = (m'/r, n'/R), m' and n' the signed frequencies; the mean mode m = n = 0 is left
// out) and writes the two sums to part[2 b], part[2 b + 1].  The twiddles are tabulated once per call instead
// of by every CTA.  1024 x 2048: 338 + 324 us for complex transforms with per-CTA twiddles, 123 + 145 us
// with real ones, 18 us less for both with butterflies of multiply-adds.  On grids
// of at most kOwnTwiddles rows and columns a CTA forms its own: a value a thread at most, less than the launch.

constexpr int kOwnTwiddles = 64;

// entry k of a per-level twiddle table
__device__ __forceinline__ C2<double> sf_twiddle(int k) {
  const int half = 1 << (31 - __clz(k + 1));  // a level's first entry is half - 1 (twiddle order of fft_strided)
  double sn, cs;
  sincospi(-(double)(k + 1 - half) / half, &sn, &cs);
  return {cs, sn};
}
__device__ __forceinline__ void sf_twiddles(C2<double>* tw, const C2<double>* table, int n) {
  if (table) return load_twiddles(tw, table, n);
  for (int k = threadIdx.x; k < n - 1; k += blockDim.x) tw[k] = sf_twiddle(k);
}

__global__ void sf_twiddle_kernel(C2<double>* tw_s, int ns, C2<double>* tw_t, int nt) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const bool first = x < ns - 1;
  const int k = first ? x : x - (ns - 1);
  if (k >= nt - 1 && !first) return;
  (first ? tw_s : tw_t)[k] = sf_twiddle(k);
}

// Rows 2 b and 2 b + 1 -> their spectra at 0 .. N_phi / 2 - 1, entry 0 holding the real values at 0 and N_phi / 2.
template <typename T>
__global__ void __launch_bounds__(256) sf_row_kernel(int ns, int logns, const T* phi, const T* phi_lo,
                                                     const C2<double>* tw_s, C2<double>* buf) {
  extern __shared__ __align__(16) unsigned char raw[];
  C2<double>* a = reinterpret_cast<C2<double>*>(raw);
  const int sh = row_pad_shift(logns), nh = ns / 2;
  C2<double>* tw = a + padded(ns, sh);
  const int64_t q = 2 * (int64_t)blockIdx.x;
  for (int s = threadIdx.x; s < ns; s += blockDim.x) {
    const int64_t g = q * ns + s, h = g + ns;
    a[padded(bitrev(s, logns), sh)] = {(double)phi[g] + (phi_lo ? (double)phi_lo[g] : 0.0),
                                       (double)phi[h] + (phi_lo ? (double)phi_lo[h] : 0.0)};
  }
  sf_twiddles(tw, tw_s, ns);
  __syncthreads();
  fft_strided(a, ns, logns, 0, sh, tw, false);
  C2<double>*r0 = buf + q * nh, *r1 = r0 + nh;
  for (int k = threadIdx.x; k < nh; k += blockDim.x) {
    const C2<double> z = a[padded(k, sh)], y = a[padded(k ? ns - k : nh, sh)];
    if (k == 0) {
      r0[0] = {z.x, y.x};
      r1[0] = {z.y, y.y};
    } else {  // (z + conj y) / 2 and (z - conj y) / 2i
      r0[k] = {0.5 * (z.x + y.x), 0.5 * (z.y - y.y)};
      r1[k] = {0.5 * (z.y + y.y), 0.5 * (y.x - z.x)};
    }
  }
}

__global__ void __launch_bounds__(256) sf_col_kernel(int nt, int lognt, int ns, int lcw, double kt, double kp,
                                                     const C2<double>* tw_t, const C2<double>* buf, double* part) {
  extern __shared__ __align__(16) unsigned char raw[];
  C2<double>* a = reinterpret_cast<C2<double>*>(raw);
  const int cw = 1 << lcw, nh = ns / 2, n0 = blockIdx.x << lcw;
  C2<double>* tw = a + ((size_t)nt << lcw);
  __shared__ double red[2][8];
  for (int idx = threadIdx.x; idx < nt << lcw; idx += blockDim.x) {
    const int q = idx >> lcw, c = idx & (cw - 1);
    a[(bitrev(q, lognt) << lcw) + c] = buf[(int64_t)q * nh + n0 + c];
  }
  sf_twiddles(tw, tw_t, nt);
  __syncthreads();
  fft_strided(a, nt, lognt, lcw, 31, tw, false);
  double s_sum = 0.0, k_sum = 0.0;
  for (int idx = threadIdx.x; idx < (nt / 2 + 1) << lcw; idx += blockDim.x) {
    const int m = idx >> lcw, c = idx & (cw - 1), n = n0 + c, mr = m ? nt - m : 0;
    const C2<double> z = a[(m << lcw) + c], y = a[(mr << lcw) + c];
    const double mk = (m * kt) * (m * kt);
    if (n) {  // columns n and N_phi - n, rows m and -m
      const double S = z.x * z.x + z.y * z.y + (mr != m ? y.x * y.x + y.y * y.y : 0.0);
      s_sum += 2.0 * S;
      k_sum += 2.0 * sqrt(mk + (n * kp) * (n * kp)) * S;
    } else {  // the packed columns 0 and N_phi / 2: (z + conj y) / 2, (z - conj y) / 2i
      const double w = mr != m ? 0.5 : 0.25;  // |.|^2 / 4, twice for the rows m and -m
      const double ax = z.x + y.x, ay = z.y - y.y, bx = z.y + y.y, by = y.x - z.x;
      const double S0 = w * (ax * ax + ay * ay), Sh = w * (bx * bx + by * by);
      if (m) {
        s_sum += S0;
        k_sum += sqrt(mk) * S0;
      }
      s_sum += Sh;
      k_sum += sqrt(mk + (nh * kp) * (nh * kp)) * Sh;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    s_sum += __shfl_xor_sync(0xffffffffu, s_sum, o);
    k_sum += __shfl_xor_sync(0xffffffffu, k_sum, o);
  }
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    red[0][warp] = s_sum;
    red[1][warp] = k_sum;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a0 = 0.0, a1 = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a0 += red[0][w];
      a1 += red[1][w];
    }
    part[2 * blockIdx.x] = a0;
    part[2 * blockIdx.x + 1] = a1;
  }
}

// columns per strip (log2): 32-byte segments of the spectrum's rows, and enough strips for every SM
int sf_strip(int nt, int ns) { return ns / 2 >= 2 && nt <= 2048 ? 1 : 0; }

}  // namespace

int structure_blocks(int nt, int ns) { return (ns / 2) >> sf_strip(nt, ns); }

template <typename T>
cudaError_t launch_structure_sums(int nt, int ns, double r, double R, const T* phi, const T* phi_lo, void* buf,
                                  double* part, cudaStream_t st) {
  if (!ch_stab_shape_ok(nt, ns)) return cudaErrorInvalidValue;
  const int lognt = ilog2(nt), logns = ilog2(ns), lcw = sf_strip(nt, ns);
  C2<double>* cb = reinterpret_cast<C2<double>*>(buf);
  C2<double>*tw_s = cb + (size_t)nt * ns / 2, *tw_t = tw_s + (ns - 1);  // (nt - 2) (ns - 2) >= 0: they fit
  if (nt <= kOwnTwiddles && ns <= kOwnTwiddles) tw_s = tw_t = nullptr;
  const size_t row_bytes = sizeof(C2<double>) * ((size_t)ns * 2 + 32);
  const size_t col_bytes = sizeof(C2<double>) * (((size_t)nt << lcw) + nt);
  constexpr size_t row_max = sizeof(C2<double>) * (4096 * 2 + 32);
  constexpr size_t col_max = sizeof(C2<double>) * 4096 * 2;
  static int m1 = 0, m2 = 0;
  cudaError_t e;
  if ((e = smem_attr(sf_row_kernel<T>, row_max, m1)) != cudaSuccess) return e;
  if ((e = smem_attr(sf_col_kernel, col_max, m2)) != cudaSuccess) return e;
  if (tw_s) {
    sf_twiddle_kernel<<<(ns + nt - 2 + 127) / 128, 128, 0, st>>>(tw_s, ns, tw_t, nt);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  sf_row_kernel<T><<<nt / 2, 256, row_bytes, st>>>(ns, logns, phi, phi_lo, tw_s, cb);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  sf_col_kernel<<<structure_blocks(nt, ns), 256, col_bytes, st>>>(nt, lognt, ns, lcw, 1.0 / r, 1.0 / R, tw_t, cb, part);
  return cudaGetLastError();
}

template cudaError_t launch_structure_sums<float>(int, int, double, double, const float*, const float*, void*,
                                                  double*, cudaStream_t);
template cudaError_t launch_structure_sums<double>(int, int, double, double, const double*, const double*, void*,
                                                   double*, cudaStream_t);

template cudaError_t launch_ch_stab<float>(int, int, double, const double*, const float*, void*, const float*,
                                           const float*, float*, int64_t, float, cudaStream_t);
template cudaError_t launch_ch_stab<double>(int, int, double, const double*, const double*, void*, const double*,
                                            const double*, double*, int64_t, double, cudaStream_t);

}  // namespace vlb
