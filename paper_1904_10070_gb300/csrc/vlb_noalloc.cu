// vlb_step_noalloc: the SSP-RK3 step without any device allocation.
//
// Some callers cannot allocate device memory at the point where they need to advance a state:
// plug-ins whose host application hands out only pre-sized device buffers from its own arena (the
// host owns the memory budget), and latency-critical loops where cudaMalloc's implicit device
// synchronisation is not acceptable.  For them this entry point keeps the two
// intermediate Runge-Kutta states and the per-row coefficient tables in one file-scope device
// array of fixed size; the caller passes only the state it owns.
//
// The array is a device symbol: host code cannot use its name as a device address.  Its address
// is obtained with cudaGetSymbolAddress once per device (with that device current) and cached.
// Every call shares the array, so two calls whose work overlaps on the GPU (different streams,
// or different host threads on one device) race; calls on one stream are ordered.  Nothing in it
// needs to start at zero: the coefficient tables are rewritten by every call, and each Runge-
// Kutta stage writes every node of its output buffer before the next stage reads it.
#include <math.h>
#include <stdio.h>

#include <mutex>

#include "vlb_node.cuh"

namespace {

constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[VLB_NOALLOC_SCRATCH_BYTES];

// Row table of the packed FP32 stages (vlb_node.cuh): they need at least 40 columns, so the scratch
// bounds their rows.  Formed in FP64 and rounded once, as the handle API forms it.
constexpr int kMaxPairRows = (int)(VLB_NOALLOC_SCRATCH_BYTES / (2 * sizeof(float) * (vlb::NARR + 1) * 40));
static __device__ __align__(256) float g_noalloc_rows[kMaxPairRows * vlb::kRowTable];
__device__ const vlb::RowRules<double> g_noalloc_rules = vlb::make_row_rules<double>();

std::mutex g_mu;
void* g_scratch_ptr[kMaxDevices] = {};
void* g_rows_ptr[kMaxDevices] = {};
thread_local char g_noalloc_err[256] = "";

// Device address of the scratch array on the current device (set-up on the first call per device).
cudaError_t scratch_address(int dev, void** out, void** rows) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&g_rows_ptr[dev], g_noalloc_rows);
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = p;
  }
  *out = g_scratch_ptr[dev];
  *rows = g_rows_ptr[dev];
  return cudaSuccess;
}

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// Row coefficient tables (the same quantities the handle API precomputes on the host), evaluated in FP64 on the
// device and rounded once to T, and with `rows` the row table.  A warp per row: lanes 0 .. 6 evaluate J at q - 2 .. q + 2
// and q +- 1/2, then a lane a coefficient, then a lane an entry, so that the chain is one sine and cosine, one
// division and a few products long (a thread per row and a second kernel for the table took 2 us more).
template <typename T>
__global__ void __launch_bounds__(64) noalloc_tables(T* coef, int nt, int nphi, int geometry, int advection, double R,
                                                     double r, float* rows, double dt, double M, double kappa) {
  const int q = (blockIdx.x * blockDim.x + threadIdx.x) / 32, k = threadIdx.x % 32;
  if (q >= nt) return;  // whole warps
  const double pi = 3.14159265358979323846;
  const double dth = 2.0 * pi / nt, dph = 2.0 * pi / nphi;
  const bool torus = geometry == VLB_TORUS;
  const double a = torus ? r / R : 0.0;
  const double off = k < 5 ? k - 2 : (k == 5 ? 0.5 : (k == 6 ? -0.5 : 0.0));
  double sn, cs;
  sincos(q * dth + off * dth, &sn, &cs);
  const double own = 1.0 + a * cs;
  auto J = [&](int lane) { return __shfl_sync(0xffffffffu, own, lane); };
  const double J0 = J(2), Jm1 = J(1), Jm2 = J(0), Jp1 = J(3), Jp2 = J(4), Jp = J(5), Jm = J(6);
  sn = __shfl_sync(0xffffffffu, sn, 2);
  double num = 1.0, den = 1.0;
  switch (k) {
    case vlb::C_J: num = J0; break;
    case vlb::C_JP: num = Jp; break;
    case vlb::C_JM: num = Jm; break;
    case vlb::C_CT: den = r * J0 * dth; break;
    case vlb::C_CP: den = R * J0 * dph; break;
    case vlb::C_GAM: num = torus ? sn : 0.0; den = R * J0; break;
    case vlb::C_LT: den = r * r * J0 * dth * dth; break;
    case vlb::C_LP: den = R * R * J0 * J0 * dph * dph; break;
    case vlb::C_GP: den = 2.0 * R * J0 * dph; break;
    case vlb::C_EP: num = -(Jm2 - 6.0 * Jm1 + 3.0 * J0 + 2.0 * Jp1) / 6.0; den = r * J0 * dth; break;
    case vlb::C_EN: num = -(-2.0 * Jm1 - 3.0 * J0 + 6.0 * Jp1 - Jp2) / 6.0; den = r * J0 * dth; break;
  }
  double c = num / den;
  const double gam = __shfl_sync(0xffffffffu, c, vlb::C_GAM);
  if (k == vlb::C_EP || k == vlb::C_EN) c = (advection == VLB_UW3 ? c : 0.0) - gam;
  if (k <= vlb::C_EN) coef[k * nt + q] = (T)c;
  if (!rows) return;
  const vlb::RowRule<double> e = g_noalloc_rules.e[k];
  const double x1 = __shfl_sync(0xffffffffu, c, e.x1), x2 = __shfl_sync(0xffffffffu, c, e.x2);
  const double y = __shfl_sync(0xffffffffu, own, e.y ? e.y - 1 : 0);
  const double s = e.s == 3 ? 1.0 : e.s == 2 ? kappa : (e.s == 1 ? dt * M : dt);
  rows[q * vlb::kRowTable + k] = vlb::row_table_entry(s * (e.c1 * x1 * (e.y ? y : 1.0) + e.c2 * x2), k);
}

const char* check_params(const vlb_params* p) {
  if (!p) return "params is NULL";
  if (p->geometry != VLB_TORUS && p->geometry != VLB_FLAT) return "geometry must be 0 or 1";
  if (p->precision != VLB_FP64 && p->precision != VLB_FP32) return "precision must be 0 or 1";
  if (p->advection != VLB_UW3 && p->advection != VLB_WENO5) return "advection must be 0 or 1";
  if (p->ch_mode != VLB_HYDRO && p->ch_mode != VLB_DIFFUSIVE) return "ch_mode must be 0 or 1";
  if (p->n_theta < (p->advection == VLB_WENO5 ? 6 : 4) || p->n_phi < 1) return "grid too small";
  if (p->n_theta > 65535 * 16) return "n_theta too large";
  if (!(p->r > 0.0) || !(p->R > 0.0) || !isfinite(p->r) || !isfinite(p->R)) return "radii must be finite and > 0";
  if (p->geometry == VLB_TORUS && !(p->R > p->r)) return "torus needs R > r";
  if (!(p->dt > 0.0) || !isfinite(p->dt) || !(p->tau > 0.0)) return "dt must be finite and > 0, tau > 0";
  if (!(p->M >= 0.0) || !(p->A >= 0.0) || !(p->kappa >= 0.0)) return "M, A, kappa must be >= 0";
  if (p->ch_stab != 0) return "the no-allocation step runs the explicit Cahn-Hilliard step (ch_stab must be 0)";
  return nullptr;
}

template <typename T>
cudaError_t run(const vlb_params* p, T* state, int64_t stride, double n0, int64_t nsteps, unsigned char* scratch,
                float* rows, cudaStream_t st) {
  const int nt = p->n_theta;
  T* coef = reinterpret_cast<T*>(scratch);
  T* U1 = reinterpret_cast<T*>(scratch + align256(sizeof(T) * vlb::NCOEF * nt));
  T* U2 = U1 + (size_t)vlb::state_arrays(sizeof(T)) * stride;
  const bool pairs = sizeof(T) == 4 && p->advection == VLB_UW3 && vlb::stage_maps_apply(nt, p->n_phi);
  noalloc_tables<T><<<(nt + 1) / 2, 64, 0, st>>>(coef, nt, p->n_phi, p->geometry, p->advection, p->R, p->r,
                                                 pairs ? rows : nullptr, p->dt, p->M, p->kappa);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  vlb::StageArgs<T> a;
  a.coef = coef;
  a.nt = nt;
  a.ns = p->n_phi;
  a.stride = stride;
  a.dt = (T)p->dt;
  a.inv_tau = (T)(1.0 / p->tau);
  a.M = (T)p->M;
  a.A = (T)p->A;
  a.kappa = (T)p->kappa;
  a.gt = (T)(1.0 / (2.0 * p->r * (2.0 * M_PI / nt)));
  a.n0 = (T)n0;
  a.err = nullptr;
  if constexpr (sizeof(T) == 4) {
    if (pairs) a.rows = rows;
  }
  for (int64_t n = 0; n < nsteps; ++n) {
    a.fin = state; a.f0 = nullptr; a.fout = U1; a.b = (T)1;
    if ((e = vlb::launch_stage<T>(a, p->advection, p->ch_mode, st)) != cudaSuccess) return e;
    a.fin = U1; a.f0 = state; a.fout = U2; a.b = (T)0.25;
    if ((e = vlb::launch_stage<T>(a, p->advection, p->ch_mode, st)) != cudaSuccess) return e;
    a.fin = U2; a.f0 = state; a.fout = state; a.b = (T)(2.0 / 3.0);
    if ((e = vlb::launch_stage<T>(a, p->advection, p->ch_mode, st)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

extern "C" {

vlb_status vlb_step_noalloc(const vlb_params* p, void* d_state, int64_t stride, double n0, int64_t nsteps,
                            void* cuda_stream, const char** error) {
  static const char* kOk = "";
  if (error) *error = kOk;
  auto fail = [&](vlb_status s, const char* msg) {
    snprintf(g_noalloc_err, sizeof g_noalloc_err, "vlb_step_noalloc: %s", msg);
    if (error) *error = g_noalloc_err;
    return s;
  };
  if (const char* why = check_params(p)) return fail(VLB_ERR_ARG, why);
  if (!d_state) return fail(VLB_ERR_ARG, "state is NULL");
  if (((uintptr_t)d_state) % 256 != 0) return fail(VLB_ERR_ARG, "state must be 256-byte aligned");
  const int64_t N = (int64_t)p->n_theta * p->n_phi;
  if (stride < N || stride % 64 != 0) return fail(VLB_ERR_ARG, "stride must be >= n_theta * n_phi and a multiple of 64");
  if (nsteps < 0) return fail(VLB_ERR_ARG, "nsteps must be >= 0");
  if (!(n0 > 0.0) || !isfinite(n0)) return fail(VLB_ERR_ARG, "n0 must be finite and > 0");
  const size_t esize = p->precision == VLB_FP64 ? 8 : 4;
  // bound the stride first, so that the size arithmetic below cannot wrap around
  const int64_t max_stride = (int64_t)(VLB_NOALLOC_SCRATCH_BYTES / (2 * (size_t)vlb::state_arrays(esize) * esize));
  if (stride > max_stride) {
    char msg[160];
    snprintf(msg, sizeof msg, "stride %lld exceeds %lld elements, the most the fixed scratch (VLB_NOALLOC_SCRATCH_BYTES) holds",
             (long long)stride, (long long)max_stride);
    return fail(VLB_ERR_ARG, msg);
  }
  const size_t need = align256(esize * vlb::NCOEF * p->n_theta) +
                      2 * (size_t)vlb::state_arrays(esize) * (size_t)stride * esize;
  if (need > VLB_NOALLOC_SCRATCH_BYTES) {
    char msg[160];
    snprintf(msg, sizeof msg, "grid needs %zu bytes of scratch, more than the fixed %zu (VLB_NOALLOC_SCRATCH_BYTES)",
             need, (size_t)VLB_NOALLOC_SCRATCH_BYTES);
    return fail(VLB_ERR_ARG, msg);
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(VLB_ERR_CUDA, cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return fail(VLB_ERR_CUDA, "device index out of range");
  void *scratch = nullptr, *rows = nullptr;
  e = scratch_address(dev, &scratch, &rows);
  if (e != cudaSuccess) return fail(VLB_ERR_CUDA, cudaGetErrorString(e));
  cudaStream_t st = (cudaStream_t)cuda_stream;
  e = esize == 8 ? run<double>(p, (double*)d_state, stride, n0, nsteps, (unsigned char*)scratch, (float*)rows, st)
                 : run<float>(p, (float*)d_state, stride, n0, nsteps, (unsigned char*)scratch, (float*)rows, st);
  if (e != cudaSuccess) return fail(VLB_ERR_CUDA, cudaGetErrorString(e));
  return VLB_OK;
}

}  // extern "C"
