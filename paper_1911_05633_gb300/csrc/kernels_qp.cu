// Linearised quasiparticle energies on the device: Sigma_c(i w) ~ S0 + i w S1 through the
// two lowest positive fermionic frequencies, then the eigenvalues of
// A^{-1} (H + Sigma_x^h + S0^h - mu) A^{-1} + mu with A = (I - S1^h)^{1/2} (h: Hermitian part).
// One block per momentum, in shared memory.
#include <cuda_runtime.h>

#include <cmath>
#include <string>

#include "dyson.h"
#include "ktimer.h"
#include "smem_limit.h"

namespace gw {

namespace {

__device__ __forceinline__ double2 conjq(double2 a) { return make_double2(a.x, -a.y); }

__device__ __forceinline__ double2 cfmq(double2 a, double2 b, double2 c) {  // c + a b
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}

// Hermitian part of element (i, j) of M (row-major N x N) at offset base.
__device__ __forceinline__ double2 herm_el(const double2* __restrict__ M, long long base, int N, int i, int j) {
  const double2 x = M[base + (long long)i * N + j], y = M[base + (long long)j * N + i];
  return make_double2(0.5 * (x.x + y.x), 0.5 * (x.y - y.y));
}

// Leading dimension in shared memory: odd, so that the words of a column fall on different banks.
__host__ __device__ inline int qp_ld(int N) { return N | 1; }
constexpr int kQT = 256;     // threads per block
// Sections of an eigenvalue's interval per step, 2^bits: as many (up to 64) as four warps have
// lanes for, four at least.  A step is a chain of N divisions, which four warps of an SM take in
// the latency of one and eight do not: N = 2 46 us with four sections, 28 with 64; N = 16 327 with
// four, 266 with eight, 311 with 16; N = 32 709 with four, 757 with eight.
__host__ __device__ constexpr int qp_bits(int N) {
  int bits = 2;
  while (bits < 6 && N * ((2 << bits) - 1) <= 128) ++bits;
  return bits;
}
static_assert(kQpMaxN * ((1 << qp_bits(kQpMaxN)) - 1) <= kQT, "one thread per section point");

// f(i, j) over the rows and columns r0 .. N - 1, flattened over the block (every lane busy:
// the FP64 pipe issues two multiply-adds per clock and SM, so idle lanes are what costs).
template <typename F>
__device__ __forceinline__ void each(int rows, int cols, F f) {
  const int di = kQT / cols, dj = kQT - di * cols;
  int i = threadIdx.x / cols, j = threadIdx.x - (threadIdx.x / cols) * cols;
  while (i < rows) {
    f(i, j);
    i += di;
    j += dj;
    if (j >= cols) { j -= cols; ++i; }
  }
}

// One block per momentum k.  The energies are the eigenvalues of X c = (E - mu) B c with
// X = H^h + Sigma_x^h + S0^h - mu and B = I - S1^h, the same as those of A^{-1} X A^{-1},
// A = B^{1/2}: B = L L^H by Cholesky, Z = L^{-1} X L^{-H}, Z to a real tridiagonal by
// Householder reflections, its eigenvalues by sections on Sturm counts (all at once, one
// thread per eigenvalue and interior point).  About 13 N^3 FP64 operations per momentum; the
// cyclic Jacobi iterations this replaces took about 270 N^3: 2.96 ms for 64 momenta of N = 72, against 34.3.
__global__ void __launch_bounds__(kQT) k_qp_energies(const double2* __restrict__ H, const double2* __restrict__ Sx,
                                                     const double2* __restrict__ Sc, int n_w, int i0, int i1,
                                                     double w0, double w1, double mu, int N,
                                                     double* __restrict__ E) {
  extern __shared__ double2 smq[];
  const int ld = qp_ld(N);
  double2* X = smq;                                   // [N][ld]
  double2* L = X + (size_t)N * ld;                    // [N][ld]
  double2* v = L + (size_t)N * ld;                    // [N] Householder vector
  double2* p = v + N;                                 // [N]
  double* d = reinterpret_cast<double*>(p + N);       // [N] diagonal
  double* e2 = d + N;                                 // [N] squared off-diagonals
  __shared__ double s_beta, s_lo, s_hi, s_min;
  __shared__ int s_on;
  __shared__ double lo[kQpMaxN], hi[kQpMaxN];
  __shared__ int above[kQpMaxN];  // first interior point with more than that many eigenvalues below it
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const long long k = blockIdx.x;
  const long long NN = (long long)N * N;
  const long long b0 = (k * n_w + i0) * NN, b1 = (k * n_w + i1) * NN;
  // S1 = (Sc(i w1) - Sc(i w0)) / (i (w1 - w0)); S0 = Sc(i w0) - i w0 S1
  const double fw = 1.0 / (w1 - w0);
  auto s1 = [&](int i, int j) -> double2 {
    if (!Sc) return make_double2(0.0, 0.0);
    const double2 d1 = Sc[b1 + (long long)i * N + j], d0 = Sc[b0 + (long long)i * N + j];
    return make_double2((d1.y - d0.y) * fw, -(d1.x - d0.x) * fw);  // (d1 - d0) / i
  };
  auto s0 = [&](int i, int j) -> double2 {
    if (!Sc) return make_double2(0.0, 0.0);
    const double2 d0 = Sc[b0 + (long long)i * N + j], m = s1(i, j);
    return make_double2(d0.x + w0 * m.y, d0.y - w0 * m.x);  // d0 - i w0 S1
  };
  each(N, N, [&](int i, int j) {
    const double2 a = s1(i, j), b = s1(j, i);
    L[i * ld + j] = make_double2((i == j ? 1.0 : 0.0) - 0.5 * (a.x + b.x), -0.5 * (a.y - b.y));
    double2 z = herm_el(H, k * NN, N, i, j);
    if (Sx) {
      const double2 y = herm_el(Sx, k * NN, N, i, j);
      z.x += y.x;
      z.y += y.y;
    }
    const double2 f = s0(i, j), q = s0(j, i);
    z.x += 0.5 * (f.x + q.x) - (i == j ? mu : 0.0);
    z.y += 0.5 * (f.y - q.y);
    X[i * ld + j] = z;
  });
  __syncthreads();
  // Cholesky, column by column (an indefinite B gives NaN energies); the reciprocal of the
  // diagonal stands on the diagonal, and X <- L^{-1} X takes its step j in the same pass
  for (int j = 0; j < N; ++j) {
    if (t == 0) L[j * ld + j] = make_double2(1.0 / sqrt(L[j * ld + j].x), 0.0);
    __syncthreads();
    const double r = L[j * ld + j].x;
    for (int i = t; i < N; i += kQT) {
      X[j * ld + i] = make_double2(r * X[j * ld + i].x, r * X[j * ld + i].y);
      if (i > j) L[i * ld + j] = make_double2(r * L[i * ld + j].x, r * L[i * ld + j].y);
    }
    __syncthreads();
    const int m = N - 1 - j;
    if (m > 0) {
      each(m, m, [&](int a, int b) {  // B_ic -= L_ij conj(L_cj), the lower triangle
        if (b > a) return;
        const double2 x = L[(j + 1 + a) * ld + j], y = L[(j + 1 + b) * ld + j];
        double2* z = L + (j + 1 + a) * ld + j + 1 + b;
        *z = cfmq(x, make_double2(-y.x, y.y), *z);
      });
      each(m, N, [&](int a, int c) {
        const double2 x = L[(j + 1 + a) * ld + j];
        double2* z = X + (j + 1 + a) * ld + c;
        *z = cfmq(make_double2(-x.x, -x.y), X[j * ld + c], *z);
      });
    }
    __syncthreads();
  }
  // Z = X L^{-H}: column j scaled, taken out of the columns after it
  for (int j = 0; j < N; ++j) {
    const double r = L[j * ld + j].x;
    for (int i = t; i < N; i += kQT) X[i * ld + j] = make_double2(r * X[i * ld + j].x, r * X[i * ld + j].y);
    __syncthreads();
    const int m = N - 1 - j;
    if (m > 0)
      each(N, m, [&](int i, int c) {
        const double2 y = L[(j + 1 + c) * ld + j];
        double2* z = X + i * ld + j + 1 + c;
        *z = cfmq(make_double2(-y.x, y.y), X[i * ld + j], *z);
      });
    __syncthreads();
  }
  // the Hermitian part, into L's storage
  each(N, N, [&](int i, int j) {
    const double2 a = X[i * ld + j], b = X[j * ld + i];
    L[i * ld + j] = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
  });
  __syncthreads();
  double2* A = L;
  for (int c = 0; c + 1 < N; ++c) {
    const int r0 = c + 1, m = N - r0;
    if (wid == 0) {
      double below = 0.0;
      for (int i = r0 + 1 + lane; i < N; i += 32) {
        const double2 z = A[i * ld + c];
        below = fma(z.x, z.x, fma(z.y, z.y, below));
        v[i] = z;
      }
      for (int o = 16; o > 0; o >>= 1) below += __shfl_xor_sync(0xffffffffu, below, o);
      if (lane == 0) {
        const double2 x0 = A[r0 * ld + c];
        const double a0 = x0.x * x0.x + x0.y * x0.y;
        d[c] = A[c * ld + c].x;
        e2[c] = below + a0;
        s_on = !(below == 0.0);
        // v = x + e^{i theta} |x| e_1, beta = 2 / v^H v
        const double norm = sqrt(below + a0), ab = sqrt(a0);
        const double2 ph = ab > 0.0 ? make_double2(x0.x / ab, x0.y / ab) : make_double2(1.0, 0.0);
        v[r0] = make_double2(fma(ph.x, norm, x0.x), fma(ph.y, norm, x0.y));
        s_beta = 1.0 / (norm * (norm + ab));
      }
    }
    __syncthreads();
    if (s_on) {
      const double beta = s_beta;
      // p = beta A v, four lanes per row
      for (int i = r0 + (t >> 2); i < N; i += kQT / 4) {
        const unsigned mask = 0xFu << (lane & ~3);
        double2 acc = make_double2(0.0, 0.0);
        for (int j = r0 + (t & 3); j < N; j += 4) acc = cfmq(A[i * ld + j], v[j], acc);
        for (int o = 1; o < 4; o <<= 1) {
          acc.x += __shfl_xor_sync(mask, acc.x, o);
          acc.y += __shfl_xor_sync(mask, acc.y, o);
        }
        if ((t & 3) == 0) p[i] = make_double2(beta * acc.x, beta * acc.y);
      }
      __syncthreads();
      if (wid == 0) {  // w = p - (beta / 2) (v^H p) v
        double g = 0.0;
        for (int i = r0 + lane; i < N; i += 32) g = fma(v[i].x, p[i].x, fma(v[i].y, p[i].y, g));
        for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
        g *= -0.5 * beta;
        for (int i = r0 + lane; i < N; i += 32) p[i] = make_double2(fma(g, v[i].x, p[i].x), fma(g, v[i].y, p[i].y));
      }
      __syncthreads();
      // A -= v w^H + w v^H
      each(m, m, [&](int a, int b) {
        const int i = r0 + a, j = r0 + b;
        const double2 vi = v[i], wi = p[i], vj = v[j], wj = p[j];
        double2* z = A + i * ld + j;
        *z = cfmq(make_double2(-wi.x, -wi.y), conjq(vj), cfmq(make_double2(-vi.x, -vi.y), conjq(wj), *z));
      });
    }
    __syncthreads();
  }
  if (t == 0) {
    d[N - 1] = A[(N - 1) * ld + N - 1].x;
    e2[N - 1] = 0.0;
  }
  __syncthreads();
  // an interval that holds every eigenvalue (Gershgorin), and the smallest pivot of a count
  if (wid == 0) {
    double a = 1e300, b = -1e300, e = 0.0;
    for (int i = lane; i < N; i += 32) {
      const double r = sqrt(e2[i]) + (i > 0 ? sqrt(e2[i - 1]) : 0.0);
      a = fmin(a, d[i] - r);
      b = fmax(b, d[i] + r);
      e = fmax(e, e2[i]);
    }
    for (int o = 16; o > 0; o >>= 1) {
      a = fmin(a, __shfl_xor_sync(0xffffffffu, a, o));
      b = fmax(b, __shfl_xor_sync(0xffffffffu, b, o));
      e = fmax(e, __shfl_xor_sync(0xffffffffu, e, o));
    }
    if (lane == 0) {
      const double pad = 4e-16 * N * fmax(fabs(a), fabs(b)) + 1e-300;
      s_lo = a - pad;
      s_hi = b + pad;
      s_min = fmax(e, 1.0) * 2.3e-308;
    }
  }
  __syncthreads();
  const int bits = qp_bits(N), points = (1 << bits) - 1;
  const double part = 1.0 / (1 << bits);
  const int ev = t / points, pt = t - ev * points;
  if (pt == 0 && ev < N) {
    lo[ev] = s_lo;
    hi[ev] = s_hi;
    above[ev] = points;
  }
  bool nan = false;
  for (int i = 0; i < N; ++i) nan = nan || !(fabs(d[i]) < 1e300) || !(e2[i] < 1e300);
  const double pmin = s_min;
  __syncthreads();
  // 2^56 sections: below the last bit of the largest eigenvalue
  for (int it = 0; it < 56; it += bits) {
    if (ev < N) {
      const double x = lo[ev] + (hi[ev] - lo[ev]) * (part * (pt + 1));
      int n = 0;  // eigenvalues below x: negative pivots of T - x
      double q = d[0] - x;
      if (fabs(q) < pmin) q = -pmin;
      n += q < 0.0;
      for (int i = 1; i < N; ++i) {
        q = d[i] - x - e2[i - 1] / q;
        if (fabs(q) < pmin) q = -pmin;
        n += q < 0.0;
      }
      if (n > ev) atomicMin(&above[ev], pt);
    }
    __syncthreads();
    if (ev < N && pt == 0) {
      // the section whose lower end has at most ev eigenvalues below it and whose upper end more
      const int s = above[ev];
      const double a = lo[ev], w = hi[ev] - lo[ev];
      lo[ev] = s > 0 ? a + w * (part * s) : a;
      if (s < points) hi[ev] = a + w * (part * (s + 1));
      above[ev] = points;
    }
    __syncthreads();
  }
  if (t < N) E[k * N + t] = nan ? __longlong_as_double(0x7ff8000000000000ll) : 0.5 * (lo[t] + hi[t]) + mu;
}

}  // namespace

gw_status qp_energies(const HostPlan& h, const double2* H, const double2* Sigx, const double2* Sigc, double mu,
                      double* E, cudaStream_t st) {
  const int N = h.n_orb_total();
  int i0 = -1, i1 = -1;
  for (int n = 0; n < h.n_omega; ++n) {
    if (h.omega_idx[n] == 0) i0 = n;
    if (h.omega_idx[n] == 1) i1 = n;
  }
  if (i0 < 0 || i1 < 0) {
    set_last_error("the sampled fermionic frequencies do not include n = 0 and n = 1");
    return GW_ERR_ARG;
  }
  if (N > kQpMaxN) {
    set_last_error("quasiparticle energies: more orbitals than the compiled limit");
    return GW_ERR_UNSUPPORTED;
  }
  const size_t smem = (2 * (size_t)N * qp_ld(N) + 2 * (size_t)N) * sizeof(double2) + 2 * (size_t)N * sizeof(double);
  cudaError_t e = raise_smem_limit(k_qp_energies, smem);
  if (e != cudaSuccess) {
    set_last_error(std::string("quasiparticle energies: ") + cudaGetErrorString(e));
    return GW_ERR_CUDA;
  }
  {
    TimedLaunch tl_("k_qp_energies", st);
    k_qp_energies<<<h.n_k, kQT, smem, st>>>(H, Sigx, Sigc, h.n_omega, i0, i1, M_PI / h.beta, 3.0 * M_PI / h.beta, mu,
                                            N, E);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_last_error(std::string("k_qp_energies: ") + cudaGetErrorString(e));
    return GW_ERR_CUDA;
  }
  return GW_OK;
}

}  // namespace gw
