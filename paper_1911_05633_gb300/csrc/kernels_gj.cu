// Dense FP64 work on batches of small complex matrices, one block per matrix held in
// shared memory: the in-place Gauss-Jordan inverse, and the reduction to Hessenberg form
// from which the trace of the inverse follows for any shift of the diagonal.
//
// GB300 issues about two FP64 multiply-adds per clock and SM (1.25 TFLOP/s measured), so
// these kernels are bound by the count of FP64 instructions, idle lanes included: the
// element updates run over the flattened matrix (every lane busy), and scalar work
// (pivots, reciprocals, norms) is done by one warp while another resident block computes.
#include <cuda_runtime.h>

#include <algorithm>

#include "gj.h"
#include "kernels.h"
#include "ktimer.h"
#include "smem_limit.h"

namespace gw {

namespace {

constexpr int kT = 256;

__device__ __forceinline__ double2 cmul_(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
// c + a b
__device__ __forceinline__ double2 cfma_(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
// c + conj(a) b
__device__ __forceinline__ double2 cfmaj_(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, fma(a.y, b.y, c.x)), fma(a.x, b.y, fma(-a.y, b.x, c.y)));
}
__device__ __forceinline__ double wsum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// |re| + |im| as a key that orders like it: comparisons of doubles run on the FP64 pipe,
// comparisons of the bits do not.  NaN: -1.
__device__ __forceinline__ long long size_key(double2 z) {
  const long long b = __double_as_longlong(fabs(z.x) + fabs(z.y));
  return b > 0x7ff0000000000000ll ? -1ll : b;
}

// Leading dimension of a matrix in shared memory: odd, so that the 16-byte words of a
// column fall on different banks.
__host__ __device__ inline int ld_odd(int N) { return N | 1; }
// Words of one matrix of the trace kernel: the row in hand, its derivative, two fresh rows.
__host__ __device__ inline int trace_stride(int N) { return 4 * N; }
__device__ __forceinline__ void copy16_async(double2* dst_smem, const double2* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst_smem)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// ---------------------------------------------------------------------------
// In-place Gauss-Jordan inverse, partial pivoting by |re| + |im| among the rows not yet
// used (the first of equal ones, rows counted in the order the exchanges of the textbook
// form would give them).  No rows move: column k is eliminated with pivot row p_k where it
// lies, and the exchanges are undone as the result is written, inv[k][p_l] = A[p_k][l].
// Two blocks per SM at N = 72.  3072 inverses of N = 72: 8.58 ms (1.07 TFLOP/s of the 1.25
// that FMA chains reach), 17.0 ms for the form that kept the matrix in global memory with
// one warp per row; 112 of N = 16: 30 us against 134 us.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kT, 2) k_gj_inverse_smem(double2* __restrict__ A, int N, long long mat_stride,
                                                           int* status) {
  extern __shared__ double2 smg[];
  const int ld = ld_odd(N);
  double2* M = smg;                                 // [N][ld]
  double2* rowk = M + (size_t)N * ld;               // [N] scaled pivot row
  double2* colk = rowk + N;                         // [N] multipliers
  int* at = reinterpret_cast<int*>(colk + N);       // [N] row at each place of the exchanged order
  int* piv = at + N;                                // [N] pivot row of each column
  __shared__ double2 s_inv;
  __shared__ int s_p;
  const int b = blockIdx.x;
  double2* G = A + (long long)b * mat_stride;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int NN = N * N;
  const int di = kT / N, dj = kT - di * N;  // advance of (i, j) per step of kT elements
  {
    int i = t / N, j = t - (t / N) * N;
    for (int x = t; x < NN; x += kT) {
      M[i * ld + j] = G[x];
      i += di;
      j += dj;
      if (j >= N) { j -= N; ++i; }
    }
  }
  for (int i = t; i < N; i += kT) at[i] = i;
  __syncthreads();
  for (int k = 0; k < N; ++k) {
    if (wid == 0) {
      long long best = -1;
      int bi = k;  // place in the exchanged order
      for (int i = k + lane; i < N; i += 32) {
        const long long m = size_key(M[at[i] * ld + k]);
        if (m > best) { best = m; bi = i; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (lane == 0) {
        const int p = at[bi];
        at[bi] = at[k];
        at[k] = p;
        piv[k] = p;
        s_p = p;
        if (best <= 0) atomicExch(status, 1);
        const double2 d = M[p * ld + k];
        const double den = fma(d.x, d.x, d.y * d.y), id = 1.0 / den;
        s_inv = den > 0.0 ? make_double2(d.x * id, -d.y * id) : make_double2(0.0, 0.0);
      }
    }
    __syncthreads();
    const int p = s_p;
    const double2 inv = s_inv;
    for (int j = t; j < N; j += kT) {
      rowk[j] = (j == k) ? inv : cmul_(M[p * ld + j], inv);
      const double2 f = M[j * ld + k];  // row j of column k
      colk[j] = make_double2(-f.x, -f.y);
    }
    __syncthreads();
    {
      int i = t / N, j = t - (t / N) * N;
      for (int x = t; x < NN; x += kT) {
        double2* m = M + i * ld + j;
        const double2 r = rowk[j];
        if (i == p) {
          *m = r;
        } else {
          const double2 z = (j == k) ? make_double2(0.0, 0.0) : *m;
          *m = cfma_(colk[i], r, z);
        }
        i += di;
        j += dj;
        if (j >= N) { j -= N; ++i; }
      }
    }
    __syncthreads();
  }
  {
    int i = t / N, j = t - (t / N) * N;
    for (int x = t; x < NN; x += kT) {
      G[(long long)i * N + piv[j]] = M[piv[i] * ld + j];
      i += di;
      j += dj;
      if (j >= N) { j -= N; ++i; }
    }
  }
}

// ---------------------------------------------------------------------------
// Householder reduction of M_b = i w_n - H(k) - Sigma_x(k) - Sigma_c(k, i w_n),
// b = k n_w + n, to upper Hessenberg form, out[b] = Q^dagger M_b Q (below the first
// subdiagonal: zeros).  tr (mu + M_b)^{-1} = tr (mu + out[b])^{-1} for every mu.
// Per column one rank-2 update A -= v u^T + t conj(v)^T over the flattened matrix; the two
// matrix-vector products before it run four lanes per dot product.  In shared memory when
// the matrix fits, else in `out` itself (through L2: 8 FP64 instructions per 16 bytes keep
// the FP64 pipe the bound).  3072 of N = 72: 18.2 ms, 13 ms of it FP64 issue.
// ---------------------------------------------------------------------------
template <bool SMEM>
__global__ void __launch_bounds__(kT) k_hessenberg(const double2* __restrict__ H, const double2* __restrict__ Sx,
                                                   const double2* __restrict__ Sc, const double* __restrict__ w,
                                                   int N, int n_w, double2* __restrict__ out,
                                                   double* __restrict__ scale) {
  extern __shared__ double2 smh[];
  __shared__ double s_beta, s_red[kT / 32];
  __shared__ int s_on;
  const long long b = blockIdx.x;
  const long long kq = b / n_w;
  const int n = (int)(b - kq * n_w);
  const int NN = N * N;
  const int ld = SMEM ? ld_odd(N) : N;
  double2* G = out + b * NN;
  double2* v = smh;      // [N] Householder vector, zero up to row k
  double2* tv = v + N;   // [N] beta A v
  double2* u = tv + N;   // [N] beta (v^dagger A - beta gamma conj(v))
  double2* A = SMEM ? u + N : G;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  {
    double big = 0.0;
    const int di = kT / N, dj = kT - di * N;
    int i = t / N, j = t - (t / N) * N;
    for (int x = t; x < NN; x += kT) {
      const double2 h = H[kq * NN + x];
      double re = -h.x, im = -h.y;
      if (Sx) {
        const double2 s = Sx[kq * NN + x];
        re -= s.x;
        im -= s.y;
      }
      if (Sc) {
        const double2 c = Sc[b * NN + x];
        re -= c.x;
        im -= c.y;
      }
      if (i == j) im += w[n];
      A[i * ld + j] = make_double2(re, im);
      big = fmax(big, fabs(re) + fabs(im));
      i += di;
      j += dj;
      if (j >= N) { j -= N; ++i; }
    }
    for (int o = 16; o > 0; o >>= 1) big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
    if (lane == 0) s_red[wid] = big;
    __syncthreads();
    if (t == 0) {
      for (int i2 = 1; i2 < kT / 32; ++i2) big = fmax(big, s_red[i2]);
      scale[b] = big;
    }
  }
  for (int k = 0; k + 2 < N; ++k) {
    const int r0 = k + 1, m = N - r0;  // rows and columns r0 .. N - 1
    if (wid == 0) {
      double below = 0.0;
      for (int i = r0 + 1 + lane; i < N; i += 32) {
        const double2 z = A[i * ld + k];
        below = fma(z.x, z.x, fma(z.y, z.y, below));
        v[i] = z;
      }
      below = wsum(below);
      for (int i = lane; i < r0; i += 32) v[i] = make_double2(0.0, 0.0);
      if (lane == 0) {
        const double2 x0 = A[r0 * ld + k];
        const double a0 = x0.x * x0.x + x0.y * x0.y;
        s_on = !(below == 0.0);
        const double norm = sqrt(below + a0), ab = sqrt(a0);
        // v = x + e^{i theta} |x| e_1, H x = -e^{i theta} |x| e_1, beta = 2 / v^dagger v
        const double2 ph = ab > 0.0 ? make_double2(x0.x / ab, x0.y / ab) : make_double2(1.0, 0.0);
        v[r0] = make_double2(fma(ph.x, norm, x0.x), fma(ph.y, norm, x0.y));
        s_beta = 1.0 / (norm * (norm + ab));
        if (s_on) A[r0 * ld + k] = make_double2(-ph.x * norm, -ph.y * norm);
      }
    }
    __syncthreads();
    if (!s_on) {  // the column has its form already
      __syncthreads();
      continue;
    }
    const double beta = s_beta;
    for (int i = r0 + 1 + t; i < N; i += kT) A[i * ld + k] = make_double2(0.0, 0.0);
    // s_j = sum_i conj(v_i) A_ij (columns r0 ..) into u, t_i = sum_j A_ij v_j (all rows) into tv
    const int g = t >> 2, q = t & 3;
    for (int d = g; d < m + N; d += kT / 4) {
      const unsigned mask = 0xFu << (lane & ~3);
      double2 acc = make_double2(0.0, 0.0);
      if (d < m) {
        const double2* a = A + r0 + d;
        for (int i = r0 + q; i < N; i += 4) acc = cfmaj_(v[i], a[(size_t)i * ld], acc);
      } else {
        const double2* a = A + (size_t)(d - m) * ld;
        for (int j = r0 + q; j < N; j += 4) acc = cfma_(a[j], v[j], acc);
      }
      for (int o = 1; o < 4; o <<= 1) {
        acc.x += __shfl_xor_sync(mask, acc.x, o);
        acc.y += __shfl_xor_sync(mask, acc.y, o);
      }
      if (q == 0) {
        if (d < m) u[r0 + d] = acc;
        else tv[d - m] = make_double2(-beta * acc.x, -beta * acc.y);
      }
    }
    __syncthreads();
    if (wid == 0) {
      // gamma = v^dagger A v = sum_j s_j v_j
      double2 gm = make_double2(0.0, 0.0);
      for (int j = r0 + lane; j < N; j += 32) gm = cfma_(u[j], v[j], gm);
      gm.x = beta * wsum(gm.x);
      gm.y = beta * wsum(gm.y);
      for (int j = r0 + lane; j < N; j += 32) {
        // -beta (s_j - beta gamma conj(v_j))
        const double2 c = cfmaj_(v[j], make_double2(-gm.x, -gm.y), u[j]);
        u[j] = make_double2(-beta * c.x, -beta * c.y);
      }
    }
    __syncthreads();
    {
      const int tot = N * m, di = kT / m, dj = kT - di * m;
      int i = t / m, j = t - (t / m) * m;
      for (int x = t; x < tot; x += kT) {
        double2* a = A + (size_t)i * ld + r0 + j;
        double2 z = cfmaj_(v[r0 + j], tv[i], *a);
        if (i >= r0) z = cfma_(v[i], u[r0 + j], z);
        *a = z;
        i += di;
        j += dj;
        if (j >= m) { j -= m; ++i; }
      }
    }
    __syncthreads();
  }
  if (SMEM) {
    const int di = kT / N, dj = kT - di * N;
    int i = t / N, j = t - (t / N) * N;
    for (int x = t; x < NN; x += kT) {
      G[x] = A[i * ld + j];
      i += di;
      j += dj;
      if (j >= N) { j -= N; ++i; }
    }
  }
}

// ---------------------------------------------------------------------------
// tr[b] = tr (mu + Hess_b)^{-1} = d/dmu log det (mu + Hess_b): LU with pivoting of
// neighbouring rows, carried with its derivative in mu.  G lanes per matrix (a warp holds
// 32 / G), because a row shrinks to one element and the scalar work per column (a
// reciprocal and two multipliers) is done by every lane of the matrix alike.  The row in
// hand and its derivative are in shared memory, the fresh rows arrive there one step ahead.  A pivot below `tiny` of the matrix's
// largest element, or a trace that is not finite, sets *flag.  3072 of N = 72: 0.34 ms per
// mu (0.48 with the rows fetched as they are needed, 0.66 with four lanes per matrix), 17 ms for the inverses it replaces.
// ---------------------------------------------------------------------------
template <int G>
__global__ void __launch_bounds__(32) k_hess_trace(const double2* __restrict__ Hs, const double* __restrict__ scale,
                                                   double mu, int N, long long n_b, double tiny,
                                                   double2* __restrict__ tr, int* __restrict__ flag) {
  extern __shared__ double2 smt[];
  const int per = blockDim.x / G;
  const long long b = (long long)blockIdx.x * per + threadIdx.x / G;
  const int q = threadIdx.x % G;
  const bool on = b < n_b;
  const double2* A = Hs + (on ? b : 0) * (long long)N * N;
  double2* r = smt + (size_t)(threadIdx.x / G) * trace_stride(N);  // [N] the row in hand
  double2* dr = r + N;                                    // [N] its derivative
  double2* fr = dr + N;                                   // [2][N] rows k + 1 and k + 2
  for (int j = q; j < N; j += G) {
    double2 a = A[j];
    if (j == 0) a.x += mu;
    r[j] = a;
    dr[j] = make_double2(j == 0 ? 1.0 : 0.0, 0.0);
    if (N > 1) copy16_async(fr + j, A + N + j);
  }
  copies_commit();
  const long long low = __double_as_longlong(tiny * (scale[on ? b : 0] + fabs(mu)));
  double2 sum = make_double2(0.0, 0.0);
  bool bad = false;
  for (int k = 0; k < N; ++k) {
    copies_wait();  // row k + 1 has landed; the copy of row k + 2 runs beside this step
    __syncwarp();
    const double2 rk = r[k], dk = dr[k];
    const bool last = k + 1 == N;
    const double2* nx = fr + (k & 1) * N;  // row k + 1
    if (k + 2 < N) {
      const double2* src = A + (long long)(k + 2) * N;
      double2* dst = fr + ((k + 1) & 1) * N;
      for (int j = k + 1 + q; j < N; j += G) copy16_async(dst + j, src + j);
    }
    copies_commit();
    const double2 hk = last ? make_double2(0.0, 0.0) : nx[k];
    // the fresh row's derivative is one at its diagonal, column k + 1: zero in column k
    const long long kh = size_key(hk), kr = size_key(rk);
    const bool fresh = kh > kr;
    const double2 p = fresh ? hk : rk, o = fresh ? rk : hk;
    const double2 dp = fresh ? make_double2(0.0, 0.0) : dk, dof = fresh ? dk : make_double2(0.0, 0.0);
    bad = bad || (fresh ? kh : kr) <= low;
    const double id = 1.0 / fma(p.x, p.x, p.y * p.y);
    const double2 inv = make_double2(p.x * id, -p.y * id);
    sum = cfma_(dp, inv, sum);
    if (last) break;
    // o -= f p with f = o_k / p_k, f' = (o'_k - f p'_k) / p_k
    const double2 f = cmul_(o, inv), mf = make_double2(-f.x, -f.y);
    const double2 df = cmul_(cfma_(mf, dp, dof), inv), mdf = make_double2(-df.x, -df.y);
    __syncwarp();  // every lane has read column k of the row in hand
    for (int j = k + 1 + q; j < N; j += G) {
      double2 a = nx[j];
      if (j == k + 1) a.x += mu;
      const double2 da = make_double2(j == k + 1 ? 1.0 : 0.0, 0.0);
      const double2 c = r[j], dc = dr[j];
      const double2 pj = fresh ? a : c, oj = fresh ? c : a;
      const double2 dpj = fresh ? da : dc, doj = fresh ? dc : da;
      r[j] = cfma_(mf, pj, oj);
      dr[j] = cfma_(mdf, pj, cfma_(mf, dpj, doj));
    }
  }
  if (on && q == 0) {
    tr[b] = sum;
    if (bad || !isfinite(sum.x) || !isfinite(sum.y)) atomicExch(flag, 1);
  }
}

size_t gj_smem_bytes(int N) {
  return ((size_t)N * ld_odd(N) + 2 * (size_t)N) * sizeof(double2) + 2 * (size_t)N * sizeof(int);
}
size_t hess_smem_bytes(int N, bool in_smem) {
  return (3 * (size_t)N + (in_smem ? (size_t)N * ld_odd(N) : 0)) * sizeof(double2);
}

}  // namespace

// The blocked form keeps a panel and its pivot rows in shared memory (kernels_fp64.cu).
static size_t gj_blocked_bytes(int N) { return (2 * (size_t)N * kGJB + N) * sizeof(double2); }
static bool gj_is_blocked(int N) { return gj_blocked_bytes(N) <= 220 * 1024; }

cudaError_t gj_setup(int N, bool columns) {
  if (N <= kGJSmemMax) return raise_smem_limit(k_gj_inverse_smem, gj_smem_bytes(N));
  if (!columns && gj_is_blocked(N)) return raise_smem_limit(k_gj_inverse_blocked, gj_blocked_bytes(N));
  const size_t bytes = 2 * (size_t)N * sizeof(double2);
  return bytes > 227 * 1024 ? cudaErrorInvalidValue : raise_smem_limit(k_gj_inverse, bytes);
}

// In shared memory wherever a matrix fits (N <= kGJSmemMax; 1.8x at N = 72 and 2.6x at 16
// over the forms below), else by panels while the panel and its pivot rows fit, else column
// by column in global memory.  The Dyson matrices take the columns: 768 of order 128 19.7 ms
// by panels and 16.1 by columns, of 192 54.6 and 47.5, of 384 372 and 345.
void gj_batch(double2* mats, int* perm, int batch, int N, long long stride, int* status, cudaStream_t st,
              bool columns) {
  if (N <= kGJSmemMax) {
    TimedLaunch tl_("k_gj_inverse_smem", st);
    k_gj_inverse_smem<<<batch, kT, gj_smem_bytes(N), st>>>(mats, N, stride, status);
  } else if (!columns && gj_is_blocked(N)) {
    TimedLaunch tl_("k_gj_inverse_blocked", st);
    k_gj_inverse_blocked<<<batch, 512, gj_blocked_bytes(N), st>>>(mats, perm, N, stride, status, nullptr);
  } else {
    TimedLaunch tl_("k_gj_inverse", st);
    k_gj_inverse<<<batch, 512, 2 * (size_t)N * sizeof(double2), st>>>(mats, perm, N, stride, status);
  }
}

constexpr int kTraceG = 8, kTraceThreads = 32, kTracePer = kTraceThreads / kTraceG;

cudaError_t hess_setup(int N) {
  const cudaError_t e = raise_smem_limit(k_hess_trace<kTraceG>, (size_t)kTracePer * trace_stride(N) * sizeof(double2));
  if (e != cudaSuccess) return e;
  return N <= kGJSmemMax ? raise_smem_limit(k_hessenberg<true>, hess_smem_bytes(N, true))
                         : raise_smem_limit(k_hessenberg<false>, hess_smem_bytes(N, false));
}

void hess_reduce(const double2* H, const double2* Sx, const double2* Sc, const double* w, int N, int n_w,
                 long long n_b, double2* out, double* scale, cudaStream_t st) {
  TimedLaunch tl_("k_hessenberg", st);
  if (N <= kGJSmemMax)
    k_hessenberg<true><<<(unsigned)n_b, kT, hess_smem_bytes(N, true), st>>>(H, Sx, Sc, w, N, n_w, out, scale);
  else
    k_hessenberg<false><<<(unsigned)n_b, kT, hess_smem_bytes(N, false), st>>>(H, Sx, Sc, w, N, n_w, out, scale);
}

void hess_trace(const double2* Hs, const double* scale, double mu, int N, long long n_b, double2* tr, int* flag,
                cudaStream_t st) {
  TimedLaunch tl_("k_hess_trace", st);
  // a pivot this far below the matrix leaves no digits in its reciprocal
  const double tiny = 1e-14;
  k_hess_trace<kTraceG><<<(unsigned)((n_b + kTracePer - 1) / kTracePer), kTraceThreads,
                          (size_t)kTracePer * trace_stride(N) * sizeof(double2), st>>>(Hs, scale, mu, N, n_b, tiny, tr, flag);
}

void gj_batch_only(double2* mats, int* perm, int batch, int N, int* status, const int* only, cudaStream_t st) {
  TimedLaunch tl_("k_gj_inverse_blocked<only>", st);
  k_gj_inverse_blocked<<<batch, 512, gj_blocked_bytes(N), st>>>(mats, perm, N, (long long)N * N, status, only);
}
cudaError_t gj_only_setup(int N) { return raise_smem_limit(k_gj_inverse_blocked, gj_blocked_bytes(N)); }

}  // namespace gw
