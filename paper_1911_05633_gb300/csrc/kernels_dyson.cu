// Eq. G_1 (Dyson equation) on the device, G(k, tau) through Appendix A's inverse
// transform, and the particle number from G(k, beta-).  Declarations in dyson.h.
#include <cuda_runtime.h>

#include <cmath>
#include <string>
#include <vector>

#include "dyson.h"
#include "gj.h"
#include "kernels.h"
#include "ktimer.h"
#include "smem_limit.h"

namespace gw {

namespace {

__device__ __forceinline__ double2 cfma_d(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}

// [(i w_n + mu) I - H(k) - Sigma_x(k) - Sigma_c(k, i w_n)] for block b = k n_w + n.
__global__ void k_dyson_build(const double2* __restrict__ H, const double2* __restrict__ Sx,
                              const double2* __restrict__ Sc, const double* __restrict__ w, double mu, int N, int n_w,
                              double2* __restrict__ M) {
  const long long b = blockIdx.x;
  const long long k = b / n_w;
  const int n = (int)(b - k * n_w);
  const long long NN = (long long)N * N;
  for (long long x = threadIdx.x; x < NN; x += blockDim.x) {
    const double2 h = H[k * NN + x];
    double re = -h.x, im = -h.y;
    if (Sx) {
      const double2 s = Sx[k * NN + x];
      re -= s.x;
      im -= s.y;
    }
    if (Sc) {
      const double2 c = Sc[b * NN + x];
      re -= c.x;
      im -= c.y;
    }
    if (x / N == x % N) {
      re += mu;
      im += w[n];
    }
    M[b * NN + x] = make_double2(re, im);
  }
}

// M1 = H + Sigma_x - mu of element x of momentum k
__device__ __forceinline__ double2 tail_m1(const double2* __restrict__ H, const double2* __restrict__ Sx, long long k,
                                           long long NN, long long x, bool diag, double mu) {
  const double2 h = H[k * NN + x];
  double2 m = make_double2(h.x - (diag ? mu : 0.0), h.y);
  if (Sx) {
    const double2 s = Sx[k * NN + x];
    m.x += s.x;
    m.y += s.y;
  }
  return m;
}

// G - 1/(i w) - M1/(i w)^2 = G + i/w + M1/w^2 (diagonal for the first term)
__device__ __forceinline__ double2 tail_rem(double2 g, double2 m1, double wn, bool diag) {
  const double iw2 = 1.0 / (wn * wn);
  return make_double2(fma(m1.x, iw2, g.x), fma(m1.y, iw2, g.y) + (diag ? 1.0 / wn : 0.0));
}

// G(k, tau_i) = sum_n T[i][n] rem(k, n) - 1/2 + M1 (2 tau_i - beta)/4; grid (k, chunk of
// 64 elements), each thread's remainders over n staged in shared memory.
__global__ void __launch_bounds__(64) k_green_tau(const double2* __restrict__ G, const double2* __restrict__ H,
                                                  const double2* __restrict__ Sx, const double* __restrict__ w,
                                                  const double2* __restrict__ T, const double* __restrict__ tau,
                                                  double beta, double mu, int N, int n_w, int n_tau,
                                                  double2* __restrict__ out) {
  extern __shared__ double2 rem[];  // [n_w][64]
  const long long k = blockIdx.x;
  const long long NN = (long long)N * N;
  const long long x = (long long)blockIdx.y * 64 + threadIdx.x;
  if (x >= NN) return;
  const bool diag = x / N == x % N;
  const double2 m1 = tail_m1(H, Sx, k, NN, x, diag, mu);
  for (int n = 0; n < n_w; ++n) rem[n * 64 + threadIdx.x] = tail_rem(G[(k * n_w + n) * NN + x], m1, w[n], diag);
  for (int i = 0; i < n_tau; ++i) {
    const double2* Ti = T + (long long)i * n_w;
    double2 acc = make_double2(0.0, 0.0);
    for (int n = 0; n < n_w; ++n) acc = cfma_d(Ti[n], rem[n * 64 + threadIdx.x], acc);
    const double f = (2.0 * tau[i] - beta) * 0.25;
    out[(k * n_tau + i) * NN + x] = make_double2(fma(m1.x, f, acc.x) - (diag ? 0.5 : 0.0), fma(m1.y, f, acc.y));
  }
}

// part[k] = Re Tr[-G(k, beta-)]: the last row of the inverse transform on the diagonal
// remainders, plus the tail at beta, -1/2 + M1 beta/4.  One block of 256 per k.
__global__ void __launch_bounds__(256) k_density_trace(const double2* __restrict__ G, const double2* __restrict__ H,
                                                       const double2* __restrict__ Sx, const double* __restrict__ w,
                                                       const double2* __restrict__ Tlast, double beta, double mu,
                                                       int N, int n_w, double* __restrict__ part) {
  __shared__ double red[8];
  const long long k = blockIdx.x;
  const long long NN = (long long)N * N;
  double acc = 0.0;
  for (int q = threadIdx.x; q < n_w * N; q += blockDim.x) {
    const int n = q / N, i = q - (q / N) * N;
    const long long x = (long long)i * N + i;
    const double2 r = tail_rem(G[(k * n_w + n) * NN + x], tail_m1(H, Sx, k, NN, x, true, mu), w[n], true);
    const double2 t = Tlast[n];
    acc += t.x * r.x - t.y * r.y;
  }
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    const long long x = (long long)i * N + i;
    acc += fma(tail_m1(H, Sx, k, NN, x, true, mu).x, 0.25 * beta, -0.5);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    part[k] = -s;
  }
}

// m1[k] = tr (H(k) + Sigma_x(k)).  One warp per k.
__global__ void __launch_bounds__(32) k_trace_m1(const double2* __restrict__ H, const double2* __restrict__ Sx, int N,
                                                 double2* __restrict__ m1) {
  const long long k = blockIdx.x, NN = (long long)N * N;
  double2 a = make_double2(0.0, 0.0);
  for (int i = threadIdx.x; i < N; i += 32) {
    const double2 m = tail_m1(H, Sx, k, NN, (long long)i * (N + 1), true, 0.0);
    a.x += m.x;
    a.y += m.y;
  }
  for (int o = 16; o > 0; o >>= 1) {
    a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
    a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
  }
  if (threadIdx.x == 0) m1[k] = a;
}

// out[0] = (s / N_k) sum_k Re Tr[-G(k, beta-)] from the traces tr[k n_w + n] of G(k, i w_n)
// (the sum that k_density_trace takes element by element), out[1] != 0 with *flag, which is
// cleared, or *status.  One block: n_k n_w terms of a few FP64 operations.
__global__ void __launch_bounds__(512) k_density_of_traces(const double2* __restrict__ tr,
                                                           const double2* __restrict__ m1,
                                                           const double* __restrict__ w,
                                                           const double2* __restrict__ Tlast, double beta, double mu,
                                                           int N, int n_w, int n_k, double spin, int* flag,
                                                           const int* status, double* __restrict__ out) {
  __shared__ double red[16];
  double acc = 0.0;
  for (int b = threadIdx.x; b < n_k * n_w; b += blockDim.x) {
    const int k = b / n_w, n = b - k * n_w;
    const double iw = 1.0 / w[n], iw2 = iw * iw;
    const double2 g = tr[b], m = m1[k], t = Tlast[n];
    const double rx = fma(fma(-mu, (double)N, m.x), iw2, g.x), ry = fma(m.y, iw2, g.y) + N * iw;
    acc += t.x * rx - t.y * ry;
  }
  for (int k = threadIdx.x; k < n_k; k += blockDim.x)
    acc += fma(fma(-mu, (double)N, m1[k].x), 0.25 * beta, -0.5 * N);
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < 16; ++i) s += red[i];
    out[0] = -spin * s / n_k;
    out[1] = *flag || *status ? 1.0 : 0.0;
    *flag = 0;
  }
}

gw_status launch_ok(const char* what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_last_error(std::string(what) + ": " + cudaGetErrorString(e));
    return GW_ERR_CUDA;
  }
  return GW_OK;
}

}  // namespace

gw_status dyson_init(DysonPlan& d, const HostPlan& h) {
  if (d.ready) return GW_OK;
  d.N = h.n_orb_total();
  d.n_w = h.n_omega;
  d.n_k = h.n_k;
  d.n_tau = h.n_tau;
  const size_t nb = (size_t)d.n_k * d.n_w;
  std::vector<double> w(d.n_w);
  for (int n = 0; n < d.n_w; ++n) w[n] = (2.0 * h.omega_idx[n] + 1.0) * M_PI / h.beta;
  auto up = [&](void** dst, const void* src, size_t bytes) -> bool {
    if (cudaMalloc(dst, bytes) != cudaSuccess) return false;
    d.bytes += bytes;
    return !src || cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice) == cudaSuccess;
  };
  const bool good = up((void**)&d.M, nullptr, nb * d.N * d.N * sizeof(double2)) &&
                    up((void**)&d.perm, nullptr, nb * d.N * sizeof(int)) &&
                    up((void**)&d.w, w.data(), w.size() * sizeof(double)) &&
                    up((void**)&d.tau, h.tau.data(), h.tau.size() * sizeof(double)) &&
                    up((void**)&d.part, nullptr, (size_t)d.n_k * sizeof(double)) &&
                    up((void**)&d.tr, nullptr, nb * sizeof(double2)) &&
                    up((void**)&d.scale, nullptr, nb * sizeof(double)) &&
                    up((void**)&d.m1, nullptr, (size_t)d.n_k * sizeof(double2)) &&
                    up((void**)&d.count, nullptr, 4 * sizeof(double));
  if (!good) {
    dyson_free(d);
    set_last_error("Dyson scratch allocation failed");
    return GW_ERR_OOM;
  }
  if ((size_t)d.n_w * 64 * sizeof(double2) > 227 * 1024 ||
      raise_smem_limit(k_green_tau, (int)((size_t)d.n_w * 64 * sizeof(double2))) != cudaSuccess) {
    dyson_free(d);
    set_last_error("Dyson transform: too many fermionic frequencies for shared memory");
    return GW_ERR_UNSUPPORTED;
  }
  if (gj_setup(d.N, true) != cudaSuccess || (d.N <= kHessMaxN && hess_setup(d.N) != cudaSuccess) ||
      cudaMemset(d.count, 0, 4 * sizeof(double)) != cudaSuccess) {
    dyson_free(d);
    set_last_error("Dyson solve: shared-memory opt-in");
    return GW_ERR_UNSUPPORTED;
  }
  if (uploads_landed() != cudaSuccess) {
    dyson_free(d);
    set_last_error("Dyson tables did not reach the device");
    return GW_ERR_CUDA;
  }
  d.ready = true;
  return GW_OK;
}

void dyson_free(DysonPlan& d) {
  void* ptrs[] = {d.M, d.perm, d.w, d.tau, d.part, d.tr, d.scale, d.m1, d.count, d.cont, d.spec};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  d = DysonPlan{};
}

gw_status dyson_solve(DysonPlan& d, const HostPlan& h, const double2* H, const double2* Sigx, const double2* Sigc,
                      double mu, int* d_status, cudaStream_t st) {
  (void)h;
  const int nb = d.n_k * d.n_w;
  {
    TimedLaunch tl_("k_dyson_build", st);
    k_dyson_build<<<nb, 256, 0, st>>>(H, Sigx, Sigc, d.w, mu, d.N, d.n_w, d.M);
  }
  gw_status s = launch_ok("k_dyson_build");
  if (s != GW_OK) return s;
  gj_batch(d.M, d.perm, nb, d.N, (long long)d.N * d.N, d_status, st, true);
  return launch_ok("k_gj_inverse");
}

gw_status dyson_to_tau(DysonPlan& d, const HostPlan& h, const double2* H, const double2* Sigx, double mu,
                       const double2* T, double2* G_tau, cudaStream_t st) {
  const long long NN = (long long)d.N * d.N;
  dim3 g((unsigned)d.n_k, (unsigned)((NN + 63) / 64));
  {
    TimedLaunch tl_("k_green_tau", st);
    k_green_tau<<<g, 64, (size_t)d.n_w * 64 * sizeof(double2), st>>>(d.M, H, Sigx, d.w, T, d.tau, h.beta, mu, d.N,
                                                                      d.n_w, d.n_tau, G_tau);
  }
  return launch_ok("k_green_tau");
}

gw_status dyson_density(DysonPlan& d, const HostPlan& h, const double2* H, const double2* Sigx, double mu,
                        const double2* Tlast, cudaStream_t st) {
  {
    TimedLaunch tl_("k_density_trace", st);
    k_density_trace<<<d.n_k, 256, 0, st>>>(d.M, H, Sigx, d.w, Tlast, h.beta, mu, d.N, d.n_w, d.part);
  }
  return launch_ok("k_density_trace");
}

gw_status dyson_search_begin(DysonPlan& d, const HostPlan& h, const double2* H, const double2* Sigx,
                             const double2* Sigc, cudaStream_t st) {
  const long long nb = (long long)h.n_k * d.n_w;
  hess_reduce(H, Sigx, Sigc, d.w, d.N, d.n_w, nb, d.M, d.scale, st);
  {
    TimedLaunch tl_("k_trace_m1", st);
    k_trace_m1<<<d.n_k, 32, 0, st>>>(H, Sigx, d.N, d.m1);
  }
  return launch_ok("k_hessenberg");
}

gw_status dyson_search_count(DysonPlan& d, const HostPlan& h, double mu, const double2* Tlast, const int* status,
                             double* n, bool* weak, cudaStream_t st) {
  hess_trace(d.M, d.scale, mu, d.N, (long long)h.n_k * d.n_w, d.tr, reinterpret_cast<int*>(d.count + 2), st);
  {
    TimedLaunch tl_("k_density_of_traces", st);
    k_density_of_traces<<<1, 512, 0, st>>>(d.tr, d.m1, d.w, Tlast, h.beta, mu, d.N, d.n_w, d.n_k, h.spin,
                                           reinterpret_cast<int*>(d.count + 2), status, d.count);
  }
  gw_status s = launch_ok("k_hess_trace");
  if (s != GW_OK) return s;
  double got[2];
  cudaError_t e = cudaMemcpyAsync(got, d.count, sizeof(got), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    set_last_error(std::string("particle number: ") + cudaGetErrorString(e));
    return GW_ERR_CUDA;
  }
  *n = got[0];
  *weak = got[1] != 0.0;
  return GW_OK;
}

}  // namespace gw
