// W solve on the tensor cores (Eq. W_1): each inverse (v(q)^-1, then (v^-1 - P)^-1) is
// computed in FP32 by Gauss-Jordan and refined, X <- X + X (I - A X) (twice, or four times
// beside an identity and for the pivots of the block inverse), with the residual I - A X
// evaluated to FP64 accuracy on tcgen05 from exact BF16 slices of A
// and X (an Ozaki-type splitting): after a power-of-two scaling per row of A and per
// column of X, every entry is a sum of slices a_s = alpha_s 2^-7(s+1), |alpha_s| <= 128,
// each exact in BF16 (k_oz_product below).  Two refinements take the FP32 inverse (error
// ~ kappa 1e-7) to ~1e-13 for kappa ~ 2e3.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "kernels.h"
#include "smem_limit.h"
#include "umma.h"
#include "fpbits.h"
#include "ozaki.h"
#include "gj.h"
#include "wtc.h"
#include "ktimer.h"

namespace gw {

namespace {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 c) {
  return make_float2(fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x)), fmaf(a.x, b.y, fmaf(a.y, b.x, c.y)));
}

// Barrier of the first n threads of the block (whole warps).
__device__ __forceinline__ void rows_barrier(int n) { asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory"); }

}  // namespace

// In-place FP32 Gauss-Jordan inverse with partial pivoting, one 512-thread block per
// matrix (N = 128, 256 or 384; from row and column Na, a multiple of kGJ32B, on the matrix is an
// identity and is left alone).  A panel of kGJ32B columns is reduced with one row per thread
// in registers: the pivot row, scaled by its warp, is the only operand that passes through
// shared memory, as broadcasts.  The registers rotate by one column per step (the loop stays
// rolled), so the column being eliminated is always v[0].  The row exchanges and the
// rank-kGJ32B update of the other columns, A[:, T] += (Pan - I[:, panel]) Prow (Prow: the
// pivot rows before the update), run per chunk of kGJ32C columns with 8 x 4 complex register
// blocks per thread.  At the end the columns are permuted back by the composite of the pivot
// swaps.  At N = 384 a block takes 3.9 M cycles: 2.5 M the update (1.8 M of FP32 FMAs; the
// paired fma.rn.f32x2 needs its operands copied and swapped and took 3.7 M), 1.0 M the panels,
// bound by the chain pivot - scaled row - update of each column (1.7 M with the panel in shared
// memory, and the same with a warp per row and shuffles).  900 matrices: 13.0 ms, 16.8 before.
// 196 matrices of order 288 in 384: 3.5 ms, 5.5 with the identity eliminated too.
template <int N>
__global__ void __launch_bounds__(512, 1)
k_gj_inverse_f32(float2* __restrict__ A, int Na, long long mat_stride, int* __restrict__ status,
                 int* __restrict__ weak) {
  constexpr int B = kGJ32B, C = kGJ32C, P = kGJ32P;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* Pan = reinterpret_cast<float2*>(smraw);  // [N][P], columns 0 .. B - 1 used
  float2* Buf = Pan + (size_t)N * P;               // Prow [B][C] / exchange staging [2B][C] / rows [16][N]
  int* pm = reinterpret_cast<int*>(Buf + gj32_buf_elems(N));  // [N] pivot row chosen for each column
  int* srcmap = pm + N;                            // [N]
  int* xdst = srcmap + N;                          // [2B]
  int* xsrc = xdst + 2 * B;                        // [2B]
  __shared__ unsigned cand_v[N / 32];  // pivot candidates of the warps: size and row
  __shared__ int cand_i[N / 32];
  __shared__ __align__(16) float2 raw_s[B], oldk_s[B], row_s[B];  // pivot row, old row k, scaled pivot row
  __shared__ int nx;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  float2* M = A + (long long)blockIdx.x * mat_stride;
  for (int k0 = 0; k0 < Na; k0 += B) {
    for (int x = tid; x < Na * B; x += 512) Pan[(x / B) * P + x % B] = M[(long long)(x / B) * N + k0 + (x % B)];
    __syncthreads();
    if (tid < Na) {  // whole warps
      float2 v[B];  // row tid; column k0 + (m + j) % B at step m
#pragma unroll
      for (int j = 0; j < B; j += 2) {
        const float4 q = *reinterpret_cast<const float4*>(Pan + tid * P + j);
        v[j] = make_float2(q.x, q.y);
        v[j + 1] = make_float2(q.z, q.w);
      }
#pragma unroll 1
      for (int m = 0; m < B; ++m) {
        const int k = k0 + m;
        // largest |Re| + |Im| at or below row k, the first of equals: its bits + 1, 0 for none
        const float a = fabsf(v[0].x) + fabsf(v[0].y);
        const unsigned key = tid >= k && a >= 0.0f ? __float_as_uint(a) + 1u : 0u;
        const unsigned wkey = __reduce_max_sync(0xffffffffu, key);
        const unsigned wbal = __ballot_sync(0xffffffffu, key == wkey);
        if (lane == 0) { cand_v[wid] = wkey; cand_i[wid] = 32 * wid + __ffs(wbal) - 1; }
        rows_barrier(Na);
        const unsigned ckey = lane < Na / 32 ? cand_v[lane] : 0u;
        const unsigned best = __reduce_max_sync(0xffffffffu, ckey);
        const unsigned cbal = __ballot_sync(0xffffffffu, ckey == best);
        const int p = best ? cand_i[__ffs(cbal) - 1] : k;
        if (tid == 0) {
          pm[k] = p;
          if (best < 2u) atomicExch(weak ? weak + blockIdx.x : status, 1);
        }
        if (wid == (p >> 5)) {
          if (tid == p) {
#pragma unroll
            for (int j = 0; j < B; j += 2)
              *reinterpret_cast<float4*>(raw_s + j) = make_float4(v[j].x, v[j].y, v[j + 1].x, v[j + 1].y);
          }
          __syncwarp();
          const float2 d = raw_s[0];
          const float den = d.x * d.x + d.y * d.y;
          const float2 inv = den > 0.0f ? make_float2(d.x / den, -d.y / den) : make_float2(0.0f, 0.0f);
          row_s[lane] = lane == 0 ? inv : cmul(raw_s[lane], inv);
        }
        if (tid == k) {
#pragma unroll
          for (int j = 0; j < B; j += 2)
            *reinterpret_cast<float4*>(oldk_s + j) = make_float4(v[j].x, v[j].y, v[j + 1].x, v[j + 1].y);
        }
        rows_barrier(Na);
        // rows k and p exchanged and every other row updated, one column to the left
        if (tid == p) {
#pragma unroll
          for (int j = 0; j < B; ++j) v[j] = oldk_s[j];
        }
        if (tid == k) {
#pragma unroll
          for (int j = 0; j < B; ++j) v[(j + B - 1) % B] = row_s[j];
        } else {
          const float2 f = make_float2(-v[0].x, -v[0].y);
          float4 q = *reinterpret_cast<const float4*>(row_s);
          const float2 last = cfma(f, make_float2(q.x, q.y), make_float2(0.0f, 0.0f));
          v[0] = cfma(f, make_float2(q.z, q.w), v[1]);
#pragma unroll
          for (int j = 2; j < B; j += 2) {
            q = *reinterpret_cast<const float4*>(row_s + j);
            v[j - 1] = cfma(f, make_float2(q.x, q.y), v[j]);
            v[j] = cfma(f, make_float2(q.z, q.w), v[j + 1]);
          }
          v[B - 1] = last;
        }
      }
      // Pan - I on the diagonal, as the update of the other columns takes it
      const int jd = tid - k0;
#pragma unroll
      for (int j = 0; j < B; j += 2) {
        if (j == jd) v[j].x -= 1.0f;
        if (j + 1 == jd) v[j + 1].x -= 1.0f;
        *reinterpret_cast<float4*>(Pan + tid * P + j) = make_float4(v[j].x, v[j].y, v[j + 1].x, v[j + 1].y);
      }
    }
    __syncthreads();
    for (int x = tid; x < Na * B; x += 512) {
      const int i = x / B, j = x % B;
      const float2 z = Pan[i * P + j];
      M[(long long)i * N + k0 + j] = make_float2(z.x + (i == k0 + j ? 1.0f : 0.0f), z.y);
    }
    // composite row exchange of this panel: new row r = old row srcmap[r]
    for (int i = tid; i < Na; i += 512) srcmap[i] = i;
    __syncthreads();
    if (wid == 0) {
      if (lane == 0)
        for (int m = 0; m < B; ++m) {
          const int k = k0 + m, p = pm[k];
          if (p != k) { const int t = srcmap[k]; srcmap[k] = srcmap[p]; srcmap[p] = t; }
        }
      __syncwarp();
      // the moved rows (at most 2B), compacted in row order
      int n = 0;
      for (int r0 = k0; r0 < Na; r0 += 32) {
        const int r = r0 + lane;
        const bool mv = srcmap[r] != r;
        const unsigned bal = __ballot_sync(0xffffffffu, mv);
        const int pos = n + __popc(bal & ((1u << lane) - 1u));
        if (mv && pos < 2 * B) { xdst[pos] = r; xsrc[pos] = srcmap[r]; }
        n += __popc(bal);
      }
      if (lane == 0) nx = min(n, 2 * B);
    }
    __syncthreads();
    const int n = nx;
    for (int c0 = 0; c0 < Na; c0 += C) {  // (whole chunks: N is a multiple of C)
      const bool has_panel = k0 >= c0 && k0 < c0 + C;
      // (a) the row exchange on this chunk's other columns, staged through shared memory
      for (int x = tid; x < n * C; x += 512) {
        const int e = x / C, j = c0 + (x % C);
        if (!(j >= k0 && j < k0 + B)) Buf[x] = M[(long long)xsrc[e] * N + j];
      }
      __syncthreads();
      for (int x = tid; x < n * C; x += 512) {
        const int e = x / C, j = c0 + (x % C);
        if (!(j >= k0 && j < k0 + B)) M[(long long)xdst[e] * N + j] = Buf[x];
      }
      __syncthreads();
      // (b) the pivot rows of this chunk before the update
      for (int x = tid; x < B * C; x += 512) Buf[x] = M[(long long)(k0 + x / C) * N + c0 + (x % C)];
      __syncthreads();
      // (c) rows i0 .. i0 + 7, columns c0 + lane + 32 q: 32 independent loads in flight per
      // thread, then 8 x 4 complex FMAs per pair of shared-memory vectors (z, pv)
      for (int i0 = 8 * wid; i0 < Na; i0 += 8 * 16) {
        float2 acc[8][4];
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[r][q] = M[(long long)(i0 + r) * N + c0 + lane + 32 * q];
        for (int m = 0; m < B; m += 2) {
          float2 pv[4], pw[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            pv[q] = Buf[m * C + lane + 32 * q];
            pw[q] = Buf[(m + 1) * C + lane + 32 * q];
          }
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const float4 z = *reinterpret_cast<const float4*>(Pan + (i0 + r) * P + m);
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[r][q] = cfma(make_float2(z.x, z.y), pv[q], acc[r][q]);
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[r][q] = cfma(make_float2(z.z, z.w), pw[q], acc[r][q]);
          }
        }
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int j = c0 + lane + 32 * q;
            if (!has_panel || !(j >= k0 && j < k0 + B)) M[(long long)(i0 + r) * N + j] = acc[r][q];
          }
      }
      __syncthreads();
    }
  }
  // undo the pivoting on the columns: new column j = old column srcmap[j], the composite
  // of the swaps (k, pm[k]) for k = N-1 down to 0
  for (int i = tid; i < Na; i += 512) srcmap[i] = i;
  __syncthreads();
  if (tid == 0)
    for (int k = Na - 1; k >= 0; --k) {
      const int p = pm[k];
      if (p != k) { const int t = srcmap[k]; srcmap[k] = srcmap[p]; srcmap[p] = t; }
    }
  __syncthreads();
  float2* rb = Buf + (size_t)wid * N;
  for (int i = wid; i < Na; i += 16) {
    float2* Mi = M + (long long)i * N;
    for (int j = lane; j < Na; j += 32) rb[j] = Mi[j];
    __syncwarp();
    for (int j = lane; j < Na; j += 32) Mi[j] = rb[srcmap[j]];
    __syncwarp();
  }
}

namespace {

using namespace umma;

constexpr uint64_t kWaitNs = 500ull * 1000ull * 1000ull;

}  // namespace

// `act` (or null), here and below: matrices b with act[b] == 0 are left out (NN elements each).
__global__ void k_to_f32(const double2* __restrict__ src, float2* __restrict__ dst, long long n, long long NN,
                         const int* __restrict__ act) {
  for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (long long)gridDim.x * blockDim.x) {
    if (act && !act[x / NN]) continue;
    const double2 z = src[x];
    dst[x] = make_float2((float)z.x, (float)z.y);
  }
}

// Scale exponents e with |x| < 2^e for every entry of a row of A (FP64) or of a column
// of X (FP32, or the unevaluated pair hi + lo), from the exponent fields alone: a normal
// x of biased exponent E has |x| < 2^(E - bias + 1).  0 for an all-zero row or column
// (subnormal entries count as zero).

// one warp per row
__global__ void k_row_exponent(const double2* __restrict__ A, int* __restrict__ eA, int N, int batch) {
  const int warps = blockDim.x >> 5;
  const long long row = (long long)blockIdx.x * warps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= (long long)batch * N) return;
  const double2* a = A + row * N;
  int m = 0;
  for (int k = lane; k < N; k += 32) m = max(m, max(exp_field(a[k].x), exp_field(a[k].y)));
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) eA[row] = m > 0 ? m - 1022 : 0;
}

// 32 columns j per block of 8 warps, each every 8th row (lo may be null): |hi|, |lo| < 2^(m - 126),
// so |hi + lo| < 2^(m - 125).  (One thread per column left most of the chip without loads in
// flight: 2.1 ms instead of 0.5 for the four calls over 900 matrices of N = 384.)
constexpr int kCE = 256;
__device__ __forceinline__ int col_max(int m) {
  __shared__ int part[8][32];
  part[threadIdx.x >> 5][threadIdx.x & 31] = m;
  __syncthreads();
  if (threadIdx.x < 32)
#pragma unroll
    for (int w = 1; w < 8; ++w) m = max(m, part[w][threadIdx.x]);
  return m;
}
__global__ void __launch_bounds__(kCE) k_col_exponent(const float2* __restrict__ hi, const float2* __restrict__ lo,
                                                      int* __restrict__ eX, int N) {
  const int b = blockIdx.y, j = blockIdx.x * 32 + (threadIdx.x & 31);
  const long long base = (long long)b * N * N + j;
  int m = 0;
  if (j < N)
#pragma unroll 4
    for (int k = threadIdx.x >> 5; k < N; k += 8) {
      const float2 h = hi[base + (long long)k * N];
      m = max(m, max(exp_field(h.x), exp_field(h.y)));
      if (lo) {
        const float2 l = lo[base + (long long)k * N];
        m = max(m, max(exp_field(l.x), exp_field(l.y)));
      }
    }
  m = col_max(m);
  if (threadIdx.x < 32 && j < N) eX[(long long)b * N + j] = m > 0 ? m - (lo ? 125 : 126) : 0;
}

// round(x 2^(7 ND - e)) for |x| < 2^e: fixed56 for eight digits, to 2^-63 for nine.
template <int ND>
__device__ __forceinline__ long long fixed_nd(double x, int e) {
  return fixed56(x, e - 7 * (ND - 8));
}
// Digit s of it from the top, |d_0| <= 128, |d_s| <= 64 after it (as next_digit; the bit below
// the cut is added instead of a half, which could carry out of 63 bits).
template <int ND>
__device__ __forceinline__ int digit_nd(long long& m, int s) {
  if (ND == 8) return next_digit(m, s);
  const int sh = 7 * (ND - 1 - s);
  const long long d = sh > 0 ? (m >> sh) + ((m >> (sh - 1)) & 1) : m;
  m -= (long long)((unsigned long long)d << sh);
  return (int)d;
}

// A operand digits.  Element (i, k) of matrix b -> kWSA digits of Re and of Im in the
// K-major tile layout, one chunk per (matrix, 128-row block, 16-wide K step) holding
// the 2 kWSA planes of 128 x 16 in the order (Re digits 0 .. kWSA-1, Im digits ...).
// One thread per (row i, 8 consecutive k): it reads 128 contiguous bytes and writes one
// 16-byte row of a core matrix per plane; the 32 lanes of a warp (i % 8, k half,
// (i / 8) % 2) fill 512 contiguous bytes of each plane.  ND digits (kWSA, or kWFine for
// the matrices beside an identity).
template <int ND>
__global__ void k_slice_A(const double2* __restrict__ A, const int* __restrict__ eA, uint16_t* __restrict__ Asl,
                          int N, long long n_total) {
  const int NKS = N / 16, NIB = N / 128;
  const long long n_thr = n_total / 8;
  for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < n_thr; x += (long long)gridDim.x * blockDim.x) {
    const int lane = (int)(x & 31);
    long long w = x >> 5;  // (b, ib, ks, row group pair)
    const int gp = (int)(w % 8); w /= 8;
    const int ks = (int)(w % NKS); w /= NKS;
    const int ib = (int)(w % NIB);
    const long long b = w / NIB;
    const int h = (lane >> 3) & 1;
    const int il = (lane & 7) + 8 * ((lane >> 4) + 2 * gp);  // row within the 128-row block
    const int i = ib * 128 + il;
    const int k0 = ks * 16 + 8 * h;
    const int e = eA[b * N + i];
    const double2* src = A + (b * N + i) * (long long)N + k0;
    long long mr[8], mi[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double2 z = src[u];
      mr[u] = fixed_nd<ND>(z.x, e);
      mi[u] = fixed_nd<ND>(z.y, e);
    }
    uint16_t* chunk = Asl + ((b * NIB + ib) * NKS + ks) * (long long)(w_achunk(ND) / 2);
    const uint32_t off = kmajor_offset(128, il, 8 * h) / 2;
#pragma unroll
    for (int s = 0; s < ND; ++s) {
      uint32_t pr[4], pi[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t r0 = digit_bf16(digit_nd<ND>(mr[2 * u], s), s), r1 = digit_bf16(digit_nd<ND>(mr[2 * u + 1], s), s);
        const uint32_t i0 = digit_bf16(digit_nd<ND>(mi[2 * u], s), s), i1 = digit_bf16(digit_nd<ND>(mi[2 * u + 1], s), s);
        pr[u] = r0 | (r1 << 16);
        pi[u] = i0 | (i1 << 16);
      }
      *reinterpret_cast<uint4*>(chunk + (0 * ND + s) * (128 * 16) + off) = make_uint4(pr[0], pr[1], pr[2], pr[3]);
      *reinterpret_cast<uint4*>(chunk + (1 * ND + s) * (128 * 16) + off) = make_uint4(pi[0], pi[1], pi[2], pi[3]);
    }
  }
}

// X operand digits.  Element X[k][j] = hi + lo of matrix b (k = reduction index; lo may
// be null) -> SX digits of Re and of Im in the K-major layout of the B operand (rows j),
// one chunk per (matrix, kWTN-column block, 16-wide K step) holding the 2 SX planes of
// kWTN x 16 in the order (Re digits, Im digits).  One thread per (column j, 8
// consecutive k); lanes (j % 8, k half, (j / 8) % 2) read 128-byte row segments and fill
// 512 contiguous bytes of each plane.
template <int SX>
__global__ void k_slice_X(const float2* __restrict__ hi, const float2* __restrict__ lo, const int* __restrict__ eX,
                          uint16_t* __restrict__ Xsl, int N, long long n_total) {
  constexpr int JG = kWTN / 16;  // 16-column groups per block
  const int NKS = N / 16, NJB = N / kWTN;
  const long long n_thr = n_total / 8;
  for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < n_thr; x += (long long)gridDim.x * blockDim.x) {
    const int lane = (int)(x & 31);
    long long w = x >> 5;  // (b, jb, ks, column group)
    const int jg = (int)(w % JG); w /= JG;
    const int ks = (int)(w % NKS); w /= NKS;
    const int jb = (int)(w % NJB);
    const long long b = w / NJB;
    const int h = (lane >> 3) & 1;
    const int jl = (lane & 7) + 8 * ((lane >> 4) + 2 * jg);  // column within the block
    const int j = jb * kWTN + jl;
    const int k0 = ks * 16 + 8 * h;
    const int e = eX[b * N + j];
    const long long o0 = (b * N + k0) * (long long)N + j;
    long long mr[8], mi[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float2 z = hi[o0 + (long long)u * N];
      mr[u] = fixed56(z.x, e);
      mi[u] = fixed56(z.y, e);
      if (lo) {  // each part rounds to 2^-56 of the column scale
        const float2 l = lo[o0 + (long long)u * N];
        mr[u] += fixed56(l.x, e);
        mi[u] += fixed56(l.y, e);
      }
    }
    uint16_t* chunk = Xsl + ((b * NJB + jb) * NKS + ks) * (long long)(wx_chunk(SX) / 2);
    const uint32_t off = kmajor_offset(kWTN, jl, 8 * h) / 2;
#pragma unroll
    for (int t = 0; t < SX; ++t) {
      uint32_t pr[4], pi[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t r0 = digit_bf16(next_digit(mr[2 * u], t), t), r1 = digit_bf16(next_digit(mr[2 * u + 1], t), t);
        const uint32_t i0 = digit_bf16(next_digit(mi[2 * u], t), t), i1 = digit_bf16(next_digit(mi[2 * u + 1], t), t);
        pr[u] = r0 | (r1 << 16);
        pi[u] = i0 | (i1 << 16);
      }
      *reinterpret_cast<uint4*>(chunk + (0 * SX + t) * (kWTN * 16) + off) = make_uint4(pr[0], pr[1], pr[2], pr[3]);
      *reinterpret_cast<uint4*>(chunk + (1 * SX + t) * (kWTN * 16) + off) = make_uint4(pi[0], pi[1], pi[2], pi[3]);
    }
  }
}

// ---- digit products on the tensor cores -------------------------------------------------
//
// One kernel for the residual R = I - A X of the refinements and for the panel products
// C = A B, C -= A B of the block inverse.  A complex product runs as a real one of twice the
// length: the Re rows are [Ar, -Ai] [Br; Bi] and the Im rows [Ai, Ar] [Br; Bi], so an output
// row (Re or Im) takes one digit plane of A and one of B per 16-wide K step (-Ai through the
// negate-A bit).  The digit products of level L = s + t (digit s of A, digit t of B) go to
// accumulator L; for digit s of A the digits t of B feed consecutive accumulators, so a run
// of up to four B planes, consecutive in shared memory, is one MMA of 64 x run columns: 11
// MMAs per K step for eight levels, at the full rate of the tensor core (36 MMAs 64 wide run
// at two thirds of it: their operand reads bound them).
//
// Exactness: the level sums over at most 512 real terms are integers in their unit
// 2^-7(L+2) up to 2^24 for L <= 5, exact in FP32 whatever rounding the tensor core applies;
// of eight levels 6 and 7 round far below 2^-52 of the scale.  With nine digits the sum has
// units of 2^-59: level 6 (unit 2^-56) passes 2^24 only if almost all of its 512 x 7 products
// have their largest size and one sign (18.9 M at worst), and then loses a unit; levels 7 and 8
// (2^-63 and 2^-70) are rounded together.  A longer reduction (N = 384: 768 terms)
// is taken in two halves: the accumulators are read out as exact 64-bit sums in units of
// 2^-52 in between.  The sum of all levels is rounded once.
constexpr int kPT = 512;          // threads: 4 warps per tensor-memory lane quadrant, 16 columns each
constexpr int kPExact = 512;      // real terms per read-out

// The integer of one level, |I| < 2^25 (the six-level residual keeps 768 terms in one sum):
// split at a multiple of 8, both parts read by adding 1.5 2^k (a float-to-integer conversion
// issues at the FP64 rate here: with eight of them per entry the read-out took as long as
// the products).
__device__ __forceinline__ int level_int(float v, float sc) {
  const float x = v * sc;
  const float y = x + 100663296.0f;                    // 1.5 2^26: x to a multiple of 8
  return 8 * (__float_as_int(y) - 0x4CC00000) + (__float_as_int((x - (y - 100663296.0f)) + 12582912.0f) - 0x4B400000);
}
// (unsigned: with the units of 2^-59 the sum runs modulo 2^64 until the identity is taken out)
template <int L, int UB>
__device__ __forceinline__ void add_level(unsigned long long& S, float v) {
  S += (unsigned long long)(long long)level_int(v, __int_as_float((127 + 7 * (L + 2)) << 23)) << (UB - 14 - 7 * L);
}
// the last two levels together, rounded to a unit (below 2^21 of them): 6 and 7 to 2^-52, 7 and
// 8 to 2^-59
template <int UB>
__device__ __forceinline__ void add_last2(unsigned long long& S, float v0, float v1) {
  const float sc = __int_as_float((127 + UB) << 23);
  S += (unsigned long long)(long long)(__float_as_int(fmaf(v0 + v1, sc, 12582912.0f)) - 0x4B400000);
}
// levels 5 .. 7 of one accumulator, rounded to nearest at 2^-52
__device__ __forceinline__ void add_tail(unsigned long long& S, float v) {
  const float x = v * 0x1p52f;
  S += (unsigned long long)(fabsf(x) < 0x1p25f ? (long long)level_int(x, 1.0f) : __float2ll_rn(x));
}
// S 2^e rounded once to FP32 (ties to even), from the bit fields; below 2^-126: zero
__device__ __forceinline__ float i2f_scaled(long long S, int e) {
  if (S == 0) return 0.0f;
  const uint32_t sign = S < 0 ? 0x80000000u : 0u;
  unsigned long long m = S < 0 ? (unsigned long long)(-S) : (unsigned long long)S;
  const int lz = __clzll((long long)m);
  m <<= lz;  // leading one at bit 63
  const uint32_t hi = (uint32_t)(m >> 32);
  const bool rest = (hi & 0x7Fu) != 0u || (uint32_t)m != 0u;  // below the half unit
  uint32_t f = hi >> 8;  // 24 bits with the leading one
  if ((hi & 0x80u) && (rest || (f & 1u))) ++f;
  int ex = 63 - lz + e;
  if (f >> 24) { f >>= 1; ++ex; }
  if (ex < -126) return __uint_as_float(sign);
  if (ex > 127) return __uint_as_float(sign | 0x7F800000u);
  return __uint_as_float(sign | ((uint32_t)(ex + 127) << 23) | (f & 0x7FFFFFu));
}

// The MMAs of one 16-wide K step.  `first`: the step's first product of each accumulator
// writes it.  TAIL: the levels 5 .. LMAX share accumulator 5 (written by the step `first5`).
template <int SX, int LMAX, bool TAIL, int TN>
__device__ __forceinline__ void product_issue_step(uint32_t tm, uint64_t da0, uint64_t dx0, bool neg, bool first,
                                                   bool first5) {
  constexpr uint32_t PA = 128 * 16 * 2, PX = TN * 16 * 2;  // bytes per A / B plane
  constexpr int LW = TAIL ? 4 : LMAX;                          // levels with an accumulator of their own
  if (TAIL) {
    const uint32_t id = neg ? idesc_bf16_f32_negA(128, TN) : idesc_bf16_f32(128, TN);
    bool fresh = first5;
#pragma unroll
    for (int t = 0; t < SX; ++t)
#pragma unroll
      for (int s = 0; s <= LMAX; ++s)
        if (s + t >= 5 && s + t <= LMAX) {
          mma_bf16(tm + 5 * TN, da0 + (uint64_t)((s * PA) >> 4), dx0 + (uint64_t)((t * PX) >> 4), id, fresh ? 0u : 1u);
          fresh = false;
        }
  }
#pragma unroll
  for (int s = 0; s <= LW; ++s) {
    const int nt = (LW - s + 1) < SX ? (LW - s + 1) : SX;
#pragma unroll
    for (int t0 = 0; t0 < nt; t0 += 256 / TN) {
      const int n = (nt - t0) < 256 / TN ? (nt - t0) : 256 / TN;
      const uint32_t id = neg ? idesc_bf16_f32_negA(128, TN * n) : idesc_bf16_f32(128, TN * n);
      // an accumulator's first product: digit 0 of A, or (levels beyond the digits of B) the
      // smallest digit of A that reaches it, with B's last digit
      const bool init = s == 0 || (s + t0 >= SX && t0 == SX - 1);
      mma_bf16(tm + (uint32_t)(s + t0) * TN, da0 + (uint64_t)((s * PA) >> 4), dx0 + (uint64_t)((t0 * PX) >> 4), id,
               (first && init) ? 0u : 1u);
    }
  }
}

// One block of 128 output rows (Re rows for blockIdx.y < M/128, else Im rows) x kWTN columns
// from the A digits s <= LMAX and SX digits of B, products with s + t <= LMAX.  kWStages
// shared-memory stages; while step kk runs, the stage of step kk - 1 is refilled with step
// kk - 1 + kWStages.  RES: R = I - A B in FP32 (R is small; FP32 keeps it to 2^-24 of itself),
// else C = A B or C -= A B in FP64; row blocks [skip0, skip1) are left alone.  TAIL: the
// levels 5 .. 7 in one accumulator, 21 narrow MMAs more per step (the residual of the second
// refinement keeps the rounding it always had: where v^-1 - P is close to singular, W~ follows
// the last bits of that residual).  A warp's 32 x
// 16 results go through shared memory, so that a store covers two rows of 16 columns.
// 264 complex 768 x 256 by 256 x 1024 products (N = 1024): 4.54 ms with float-to-integer
// conversions on four warps; N = 384 residuals, 900 matrices, eight levels: 7.1 ms.
template <int SX, int LMAX, bool RES, bool TAIL, int ND>
__global__ void __launch_bounds__(kPT, 1) k_oz_product(const __grid_constant__ OzProductArgs g) {
  constexpr int NL = LMAX + 1;
  constexpr int TN = w_tn(LMAX);         // columns per block
  constexpr int W = TN / 4;              // columns per warp
  constexpr int UB = NL == 9 ? 59 : 52;  // sums in units of 2^-UB
  static_assert((NL == 9 && SX == 9 && RES) || (NL == 8 && SX == 8) || (NL == 6 && SX == 5), "the level read-out below");
  static_assert(!TAIL || NL == 8, "levels 5 .. 7");
  static_assert(NL * TN <= 512, "the accumulators fit the tensor memory");
  constexpr uint32_t PA = 128 * 16 * 2, PX = TN * 16 * 2;
  constexpr uint32_t AB = NL * PA, XB = SX * PX, SB = AB + XB;  // bytes per stage
  constexpr uint32_t XC = wx_chunk(SX, TN);
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint32_t tmem_base;
  __shared__ __align__(8) uint64_t full[kWStages];
  __shared__ __align__(8) uint64_t mmad[kWStages];
  __shared__ __align__(8) uint64_t gdone;
  const int jb = blockIdx.x;
  const int NKS = g.K / 16, NIB = g.M / 128, NJB = g.Nc / TN;
  const bool imrow = (int)blockIdx.y >= NIB;
  const int ib = imrow ? (int)blockIdx.y - NIB : (int)blockIdx.y;
  if (!RES && ib >= g.skip0 && ib < g.skip1) return;  // the whole block: before any barrier or allocation
  const long long b = blockIdx.z;
  if (RES && g.act && !g.act[b]) return;
  const int NK2 = 2 * NKS;
  const int n_groups = (2 * g.K > kPExact && NL > 6) ? 2 : 1;  // six levels need no exact last bits
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int* status = g.status;
  if (warp == 0) {
    tmem_alloc(&tmem_base, 512);
    tmem_relinquish();
  }
  if (tid == 0) {
    for (int s = 0; s < kWStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&mmad[s], 1);
    }
    mbar_init(&gdone, 1);
    fence_mbar_init();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tm = tmem_base;
  const unsigned char* Abase =
      reinterpret_cast<const unsigned char*>(g.Asl) + ((b * NIB + ib) * NKS) * (long long)w_achunk(ND);
  const unsigned char* Xbase = reinterpret_cast<const unsigned char*>(g.Bsl) + ((b * NJB + jb) * NKS) * (long long)XC;
  // step kk: half 0 takes (Ar | Ai for Im rows) with Br, half 1 (Ai negated | Ar) with Bi
  auto load = [&](int kk, int st) {
    const int half = kk >= NKS ? 1 : 0, ks = kk - half * NKS;
    const int cA = imrow ? 1 - half : half;
    unsigned char* dst = sm + st * SB;
    mbar_arrive_expect_tx(&full[st], SB);
    bulk_g2s(dst, Abase + (long long)ks * w_achunk(ND) + (long long)cA * ND * PA, AB, &full[st]);
    bulk_g2s(dst + AB, Xbase + (long long)ks * XC + (long long)half * SX * PX, XB, &full[st]);
  };
  const int quad = warp & 3, c0 = W * (warp >> 2);  // this warp's lanes 32 quad .. and columns c0 ..
  const uint32_t t_addr = tm + ((uint32_t)(32 * quad) << 16) + (uint32_t)c0;
  unsigned long long S[W];
#pragma unroll
  for (int c = 0; c < W; ++c) S[c] = 0;
  bool ok = true;
  if (tid == 0)
    for (int s = 0; s < kWStages && s < NK2; ++s) load(s, s);
  for (int grp = 0; grp < n_groups; ++grp) {
    if (tid == 0 && ok) {
      const uint32_t s0 = smem_u32(sm);
      const int k_end = n_groups == 1 ? NK2 : NKS * (grp + 1);
      const int k_begin = NKS * grp;
      for (int kk = k_begin; kk < k_end; ++kk) {
        const int st = kk % kWStages;
        if (!mbar_wait(&full[st], (uint32_t)(kk / kWStages) & 1u, kWaitNs, status)) { ok = false; break; }
        fence_after_sync();
        product_issue_step<SX, LMAX, TAIL, TN>(tm, smem_desc(s0 + st * SB, 128, 256),
                                           smem_desc(s0 + st * SB + AB, 128, 256), !imrow && kk >= NKS, kk == k_begin,
                                           kk == 0);
        mma_commit(&mmad[st]);
        if (kk >= 1 && kk - 1 + kWStages < NK2) {
          // the products of step kk - 1 are done once its commit arrives: refill its stage
          const int so = (kk - 1) % kWStages;
          if (!mbar_wait(&mmad[so], (uint32_t)((kk - 1) / kWStages) & 1u, kWaitNs, status)) { ok = false; break; }
          load(kk - 1 + kWStages, so);
        }
      }
      mma_commit(&gdone);  // also on a failure: the products issued so far
      if (!ok) atomicExch(status, 2);
    }
    __syncwarp();
    const bool done = mbar_wait(&gdone, (uint32_t)grp & 1u, kWaitNs, status);
    ok = __syncthreads_and(ok && done ? 1 : 0) != 0;
    fence_after_sync();
    if (!ok) break;
    float v[32];
    if constexpr (W == 8) {  // nine levels of 32 columns
      tmem_ld8x4(t_addr, TN, v);
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        add_level<0, UB>(S[c], v[c]);
        add_level<1, UB>(S[c], v[8 + c]);
        add_level<2, UB>(S[c], v[16 + c]);
        add_level<3, UB>(S[c], v[24 + c]);
      }
      tmem_ld8x4(t_addr + 4 * TN, TN, v);
      float v8[32];
      tmem_ld8x4(t_addr + 5 * TN, TN, v8);  // the last of them is level 8
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        add_level<4, UB>(S[c], v[c]);
        add_level<5, UB>(S[c], v[8 + c]);
        add_level<6, UB>(S[c], v[16 + c]);
        add_last2<UB>(S[c], v[24 + c], v8[24 + c]);
      }
    } else {
      tmem_ld16x2(t_addr, TN, v);
#pragma unroll
      for (int c = 0; c < 16; ++c) { add_level<0, UB>(S[c], v[c]); add_level<1, UB>(S[c], v[16 + c]); }
      tmem_ld16x2(t_addr + 2 * TN, TN, v);
#pragma unroll
      for (int c = 0; c < 16; ++c) { add_level<2, UB>(S[c], v[c]); add_level<3, UB>(S[c], v[16 + c]); }
      tmem_ld16x2(t_addr + 4 * TN, TN, v);
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        add_level<4, UB>(S[c], v[c]);
        if (!TAIL) add_level<5, UB>(S[c], v[16 + c]);
        else if (grp + 1 == n_groups) add_tail(S[c], v[16 + c]);
      }
      if (NL == 8 && !TAIL) {
        tmem_ld16x2(t_addr + 6 * TN, TN, v);
#pragma unroll
        for (int c = 0; c < 16; ++c) add_last2<UB>(S[c], v[c], v[16 + c]);
      }
    }
    if (grp + 1 < n_groups) {  // the next half writes the accumulators
      fence_before_sync();
      __syncthreads();
      fence_after_sync();
    }
  }
  if (!ok) {
    if (tid == 0) atomicExch(status, 2);
  } else {
    const int i = ib * 128 + 32 * quad + lane;
    const int ea = g.eA[b * g.M + i];
    const int* eb = g.eB + b * g.Nc + jb * TN + c0;
    const int cc = lane % W, r2 = lane / W;
    constexpr int RP = 32 / W;  // rows per store
    // every product has read its stage: the stages are free for the results
    if (RES) {
      float* stg = reinterpret_cast<float*>(sm) + warp * (32 * (W + 1));
      bool range_ok = true;
      unsigned big = 0u;
#pragma unroll
      for (int c = 0; c < W; ++c) {
        const int j = jb * TN + c0 + c;
        const int e = ea + eb[c];  // (A X)_ij = 2^e sum
        unsigned long long val = S[c];
        if (!imrow && i == j) {
          if (e < -10 || e > UB) range_ok = false;
          else if (UB - e < 64) val -= 1ull << (UB - e);  // 1 = 2^(UB - e) units of 2^(e - UB)
        }
        if (e < -126 || e > 126) range_ok = false;
        const float res = i2f_scaled(-(long long)val, min(max(e, -126), 126) - UB);
        big = max(big, __float_as_uint(fabsf(res)));
        stg[lane * (W + 1) + c] = res;
      }
      __syncwarp();
      float* Rw = reinterpret_cast<float*>(g.R + (b * g.M + ib * 128 + 32 * quad) * (long long)g.Nc) + (imrow ? 1 : 0);
#pragma unroll
      for (int t = 0; t < W; ++t) {
        const int rr = RP * t + r2;
        Rw[2 * ((long long)rr * g.Nc + jb * TN + c0 + cc)] = stg[rr * (W + 1) + cc];
      }
      if (!range_ok) {  // scale outside the FP32 exponent range
        if (g.weak) g.weak[b] = 1;
        else atomicExch(status, 4);
      }
      if (g.rmax) {
        for (int o = 16; o > 0; o >>= 1) big = max(big, __shfl_xor_sync(0xffffffffu, big, o));
        if (lane == 0) atomicMax(g.rmax + b, big);
      }
    } else {
      double* stg = reinterpret_cast<double*>(sm) + warp * (32 * (W + 1));
      double* Cw = reinterpret_cast<double*>(g.C + b * g.c_ms + (long long)(ib * 128 + 32 * quad) * g.ldc) + (imrow ? 1 : 0);
      // the old C values first: independent loads in flight while the sums are rounded
      double cold[16];
#pragma unroll
      for (int t = 0; t < 16; ++t)
        cold[t] = g.accumulate ? Cw[2 * ((long long)(2 * t + r2) * g.ldc + jb * TN + c0 + cc)] : 0.0;
#pragma unroll
      for (int c = 0; c < 16; ++c) stg[lane * (W + 1) + c] = i2d_scaled((long long)S[c], ea + eb[c] - 52);
      __syncwarp();
#pragma unroll
      for (int t = 0; t < 16; ++t) {
        const int rr = 2 * t + r2;
        const double pv = stg[rr * (W + 1) + cc];
        Cw[2 * ((long long)rr * g.ldc + jb * TN + c0 + cc)] = g.accumulate ? cold[t] - pv : pv;
      }
    }
  }
  fence_before_sync();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tm, 512);
}

// Three BF16 terms of an FP32 value, v = hi + mid + lo to 2^-24 of |v| (each
// remainder is exact in FP32); bits of term s.
__device__ __forceinline__ void split3_bits(float v, uint32_t* t) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  const float r1 = v - __bfloat162float(h);
  const __nv_bfloat16 m = __float2bfloat16_rn(r1);
  const float r2 = r1 - __bfloat162float(m);
  const __nv_bfloat16 l = __float2bfloat16_rn(r2);
  t[0] = __bfloat16_as_ushort(h);
  t[1] = __bfloat16_as_ushort(m);
  t[2] = __bfloat16_as_ushort(l);
}

// 8 consecutive K elements of one operand row -> one 16-byte core-matrix row in each of
// the 6 planes (term s, Re/Im) of a kRefChunk chunk.
__device__ __forceinline__ void split3_store8(const float2* z, uint16_t* chunk, uint32_t off) {
  uint32_t tr[8][3], ti[8][3];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    split3_bits(z[u].x, tr[u]);
    split3_bits(z[u].y, ti[u]);
  }
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    uint4 pr, pi;
    pr.x = tr[0][s] | (tr[1][s] << 16); pr.y = tr[2][s] | (tr[3][s] << 16);
    pr.z = tr[4][s] | (tr[5][s] << 16); pr.w = tr[6][s] | (tr[7][s] << 16);
    pi.x = ti[0][s] | (ti[1][s] << 16); pi.y = ti[2][s] | (ti[3][s] << 16);
    pi.z = ti[4][s] | (ti[5][s] << 16); pi.w = ti[6][s] | (ti[7][s] << 16);
    *reinterpret_cast<uint4*>(chunk + (s * 2 + 0) * (128 * 16) + off) = pr;
    *reinterpret_cast<uint4*>(chunk + (s * 2 + 1) * (128 * 16) + off) = pi;
  }
}

// BF16x3 operand planes of a row-major FP32 complex matrix M[b][r][k] (rows r = the MMA's
// M or N rows, k = reduction index): one kRefChunk chunk per (matrix, 128-row block,
// 16-wide K step).  Thread mapping as in k_slice_A.
__global__ void k_split3_rows(const float2* __restrict__ M, uint16_t* __restrict__ P, int N, long long n_total,
                              const int* __restrict__ act) {
  const int NKS = N / 16, NRB = N / 128;
  const long long n_thr = n_total / 8;
  for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < n_thr; x += (long long)gridDim.x * blockDim.x) {
    const int lane = (int)(x & 31);
    long long w = x >> 5;
    const int gp = (int)(w % 8); w /= 8;
    const int ks = (int)(w % NKS); w /= NKS;
    const int rb = (int)(w % NRB);
    const long long b = w / NRB;
    if (act && !act[b]) continue;
    const int h = (lane >> 3) & 1;
    const int rl = (lane & 7) + 8 * ((lane >> 4) + 2 * gp);
    const float2* src = M + (b * N + rb * 128 + rl) * (long long)N + ks * 16 + 8 * h;
    float2 z[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) z[u] = src[u];
    split3_store8(z, P + ((b * NRB + rb) * NKS + ks) * (long long)(kRefChunk / 2), kmajor_offset(128, rl, 8 * h) / 2);
  }
}

// The same planes for the transpose: element M[b][k][r] goes to row r (for the B operand
// of X R, whose rows are the columns of R).  Thread mapping as in k_slice_X.
__global__ void k_split3_cols(const float2* __restrict__ M, uint16_t* __restrict__ P, int N, long long n_total,
                              const int* __restrict__ act) {
  const int NKS = N / 16, NRB = N / 128;
  const long long n_thr = n_total / 8;
  for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < n_thr; x += (long long)gridDim.x * blockDim.x) {
    const int lane = (int)(x & 31);
    long long w = x >> 5;
    const int gp = (int)(w % 8); w /= 8;
    const int ks = (int)(w % NKS); w /= NKS;
    const int rb = (int)(w % NRB);
    const long long b = w / NRB;
    if (act && !act[b]) continue;
    const int h = (lane >> 3) & 1;
    const int rl = (lane & 7) + 8 * ((lane >> 4) + 2 * gp);
    const float2* src = M + (b * N + ks * 16 + 8 * h) * (long long)N + rb * 128 + rl;
    float2 z[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) z[u] = src[(long long)u * N];
    split3_store8(z, P + ((b * NRB + rb) * NKS + ks) * (long long)(kRefChunk / 2), kmajor_offset(128, rl, 8 * h) / 2);
  }
}

// D = X R for one 128 x 128 tile per block (512 threads) on tcgen05, from the BF16x3
// planes of X (A operand, rows i) and of R (B operand, rows j = columns of R): the six
// term products with s + t <= 2 for each of Re = Xr Rr - Xi Ri and Im = Xr Ri + Xi Rr,
// accumulated in FP32 in two 128-column tensor-memory accumulators.  R is small, so the
// product is needed to 2^-24 of itself only.  kRefStages shared-memory stages; while step
// ks runs, the stage of step ks - 1 is refilled with step ks - 1 + kRefStages.
//   MODE 0: lo[b] = D (X1 = X0 + lo is kept as the unevaluated FP32 pair)
//   MODE 1: out[b] = hi + lo + D in FP64
//   MODE 2: out[b] += D (a further refinement of the FP64 inverse in out)
// The result leaves through 16 warps: with 4 the loads of hi and lo and the FP64 stores waited
// out their latency, 4.85 ms for 936 matrices of N = 384 whose products take 1.1.
template <int MODE>
__global__ void __launch_bounds__(kPT, 1)
k_refine_tc(const uint16_t* __restrict__ PX, const uint16_t* __restrict__ PR, const float2* __restrict__ hi,
            float2* __restrict__ lo, double2* __restrict__ out, int N, int* status, const int* __restrict__ act) {
  if (act && !act[blockIdx.z]) return;
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint32_t tmem_base;
  __shared__ __align__(8) uint64_t full[kRefStages];
  __shared__ __align__(8) uint64_t mmad[kRefStages];
  const int jb = blockIdx.x, ib = blockIdx.y;
  const long long b = blockIdx.z;
  const int NKS = N / 16, NRB = N / 128;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) {
    tmem_alloc(&tmem_base, 256);
    tmem_relinquish();
  }
  if (tid == 0) {
    for (int s = 0; s < kRefStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&mmad[s], 1);
    }
    fence_mbar_init();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tm = tmem_base;
  const unsigned char* Abase = reinterpret_cast<const unsigned char*>(PX) + ((b * NRB + ib) * NKS) * (long long)kRefChunk;
  const unsigned char* Bbase = reinterpret_cast<const unsigned char*>(PR) + ((b * NRB + jb) * NKS) * (long long)kRefChunk;
  constexpr uint32_t SB = 2 * kRefChunk;  // bytes per stage
  constexpr uint32_t PL = 128 * 16 * 2;   // bytes per plane
  bool ok = true;
  if (tid == 0) {
    const uint32_t id = idesc_bf16_f32(128, 128), idn = idesc_bf16_f32_negA(128, 128);
    const uint32_t s0 = smem_u32(sm);
    for (int s = 0; s < kRefStages && s < NKS; ++s) {
      mbar_arrive_expect_tx(&full[s], SB);
      bulk_g2s(sm + s * SB, Abase + (long long)s * kRefChunk, kRefChunk, &full[s]);
      bulk_g2s(sm + s * SB + kRefChunk, Bbase + (long long)s * kRefChunk, kRefChunk, &full[s]);
    }
    for (int ks = 0; ks < NKS; ++ks) {
      const int st = ks % kRefStages;
      if (!mbar_wait(&full[st], (uint32_t)(ks / kRefStages) & 1u, kWaitNs, status)) { ok = false; break; }
      fence_after_sync();
      const uint64_t da0 = smem_desc(s0 + st * SB, 128, 256), db0 = smem_desc(s0 + st * SB + kRefChunk, 128, 256);
      bool first = ks == 0;
#pragma unroll
      for (int sa = 0; sa < 3; ++sa) {
#pragma unroll
        for (int sb = 0; sb < 3; ++sb) {
          if (sa + sb <= 2) {
            const uint64_t dar = da0 + (uint64_t)(((sa * 2 + 0) * PL) >> 4), dai = da0 + (uint64_t)(((sa * 2 + 1) * PL) >> 4);
            const uint64_t dbr = db0 + (uint64_t)(((sb * 2 + 0) * PL) >> 4), dbi = db0 + (uint64_t)(((sb * 2 + 1) * PL) >> 4);
            const uint32_t acc = first ? 0u : 1u;
            mma_bf16(tm, dar, dbr, id, acc);          // Re += Xr Rr
            mma_bf16(tm, dai, dbi, idn, 1u);          // Re -= Xi Ri
            mma_bf16(tm + 128, dar, dbi, id, acc);    // Im += Xr Ri
            mma_bf16(tm + 128, dai, dbr, id, 1u);     // Im += Xi Rr
            first = false;
          }
        }
      }
      mma_commit(&mmad[st]);
      if (ks >= 1 && ks - 1 + kRefStages < NKS) {
        const int so = (ks - 1) % kRefStages;
        if (!mbar_wait(&mmad[so], (uint32_t)((ks - 1) / kRefStages) & 1u, kWaitNs, status)) { ok = false; break; }
        const int kn = ks - 1 + kRefStages;
        mbar_arrive_expect_tx(&full[so], SB);
        bulk_g2s(sm + so * SB, Abase + (long long)kn * kRefChunk, kRefChunk, &full[so]);
        bulk_g2s(sm + so * SB + kRefChunk, Bbase + (long long)kn * kRefChunk, kRefChunk, &full[so]);
      }
    }
  }
  const int last = NKS - 1;
  const bool done = ok && mbar_wait(&mmad[last % kRefStages], (uint32_t)(last / kRefStages) & 1u, kWaitNs, status);
  ok = __syncthreads_and(done ? 1 : 0) != 0;
  fence_after_sync();
  if (!ok) {
    if (tid == 0) atomicExch(status, 2);
  } else {
    const int quad = warp & 3, c0 = 32 * (warp >> 2);
    const uint32_t t_addr = tm + ((uint32_t)(32 * quad) << 16) + (uint32_t)c0;
    // The pipeline stages are free now: each warp stages its 32 rows x 32 columns there,
    // so that its loads and stores run along rows (32 consecutive columns per instruction).
    float2* stg = reinterpret_cast<float2*>(sm) + warp * (32 * 33);
    const long long row0 = (b * N + ib * 128 + 32 * quad) * (long long)N + jb * 128 + c0 + lane;
    {
      float re[32], im[32];
      tmem_ld16x2(t_addr, 16, re);
      tmem_ld16x2(t_addr + 128, 16, im);
#pragma unroll
      for (int c = 0; c < 32; ++c) stg[lane * 33 + c] = make_float2(re[c], im[c]);
    }
    __syncwarp();
#pragma unroll 8
    for (int rr = 0; rr < 32; ++rr) {
      const float2 z = stg[rr * 33 + lane];
      const long long o = row0 + (long long)rr * N;
      if (MODE == 1) {
        const float2 h = hi[o], l = lo[o];
        out[o] = make_double2(f2d(h.x) + f2d(l.x) + f2d(z.x), f2d(h.y) + f2d(l.y) + f2d(z.y));
      } else if (MODE == 2) {
        const double2 x = out[o];
        out[o] = make_double2(x.x + f2d(z.x), x.y + f2d(z.y));
      } else {
        lo[o] = z;
      }
    }
  }
  fence_before_sync();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tm, 256);
}

// flag[b] = 1 where the largest residual of matrix b is above `most` (one that is no number
// counts as large); else 0 with `clear`, or as it was.
__global__ void k_mark(unsigned* __restrict__ rmax, int* __restrict__ flag, int batch, float most, int clear) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= batch) return;
  if (rmax[b] > __float_as_uint(most)) flag[b] = 1;
  else if (clear) flag[b] = 0;
  rmax[b] = 0u;
}

// A back from its digits (to 2^-64 of its row's largest element, under the rounding that an
// FP64 elimination commits) for the matrices marked weak.
__global__ void k_unslice_A(const uint16_t* __restrict__ Asl, const int* __restrict__ eA, const int* __restrict__ weak,
                            double2* __restrict__ A, int N) {
  const long long b = blockIdx.y;
  if (!weak[b]) return;
  const int NKS = N / 16, NIB = N / 128;
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N * N; x += gridDim.x * blockDim.x) {
    const int i = x / N, k = x - i * N;
    const uint16_t* chunk = Asl + ((b * NIB + i / 128) * NKS + k / 16) * (long long)(w_achunk(kWFine) / 2) +
                            kmajor_offset(128, i % 128, k % 16) / 2;
    const int e = eA[b * N + i];
    double z[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      unsigned long long m = 0;
#pragma unroll
      for (int s = 0; s < kWFine; ++s) {
        const float d = __uint_as_float((uint32_t)chunk[(c * kWFine + s) * (128 * 16)] << 16);
        m += (unsigned long long)(long long)__float2int_rn(d * __int_as_float((127 + 7 * (s + 1)) << 23)) << (56 - 7 * s);
      }
      z[c] = scalbn((double)(long long)m, e - 63);
    }
    A[b * N * N + x] = make_double2(z[0], z[1]);
  }
}

__global__ void k_panel_col_exp(const double2* __restrict__ B, long long ms, int ld, int K, int Nc,
                                int* __restrict__ e, const int* __restrict__ act);
template <int ND>
__global__ void k_slice_panel_B(const double2* __restrict__ B, long long ms, int ld, const int* __restrict__ eB,
                                uint16_t* __restrict__ Bsl, int K, int Nc, long long n_thr,
                                const int* __restrict__ act);

cudaError_t wtc_setup() {
  cudaError_t e = raise_smem_limit(k_gj_inverse_f32<128>, gj32_smem(128));
  if (e == cudaSuccess) e = raise_smem_limit(k_gj_inverse_f32<256>, gj32_smem(256));
  if (e == cudaSuccess) e = raise_smem_limit(k_gj_inverse_f32<384>, gj32_smem(384));
  if (e == cudaSuccess) e = raise_smem_limit(k_oz_product<kWSX0, kWL0, true, false, kWSA>, w_residual_smem(kWSX0, kWL0));
  if (e == cudaSuccess) e = raise_smem_limit(k_oz_product<kWSX1, kWLmax, true, true, kWSA>, w_residual_smem(kWSX1, kWLmax));
  if (e == cudaSuccess) e = raise_smem_limit(k_oz_product<kWSX1, kWLmax, true, false, kWSA>, w_residual_smem(kWSX1, kWLmax));
  if (e == cudaSuccess) e = raise_smem_limit(k_oz_product<kWSX0, kWL0, true, false, kWFine>, w_residual_smem(kWSX0, kWL0));
  if (e == cudaSuccess)
    e = raise_smem_limit(k_oz_product<kWSX1, kWLmax, true, true, kWFine>, w_residual_smem(kWSX1, kWLmax));
  if (e == cudaSuccess)
    e = raise_smem_limit(k_oz_product<kWFine, kWFine - 1, true, false, kWFine>, w_residual_smem(kWFine, kWFine - 1));
  if (e == cudaSuccess) e = raise_smem_limit(k_refine_tc<0>, w_refine_smem());
  if (e == cudaSuccess) e = raise_smem_limit(k_refine_tc<1>, w_refine_smem());
  if (e == cudaSuccess) e = raise_smem_limit(k_refine_tc<2>, w_refine_smem());
  return e;
}

void wtc_inverse(const WtcBuffers& w, double2* mats, int batch, int N, cudaStream_t st, int refinements, int n) {
  const long long NN = (long long)N * N;
  const int Na = n > 0 ? (n + kGJ32B - 1) / kGJ32B * kGJ32B : N;
  const bool fine = w.weak != nullptr;
  const long long tot = (long long)batch * NN;
  const unsigned g1 = (unsigned)((tot + 255) / 256 < 65535LL * 8 ? (tot + 255) / 256 : 65535LL * 8);
  const long long t8 = tot / 8;  // slicing threads: one per 8 consecutive elements
  const unsigned g8 = (unsigned)((t8 + 255) / 256 < 65535LL * 8 ? (t8 + 255) / 256 : 65535LL * 8);
  const dim3 gcol((unsigned)((N + 31) / 32), (unsigned)batch);
  const dim3 gres((unsigned)(N / kWTN), (unsigned)(2 * (N / 128)), (unsigned)batch);  // Re rows, then Im rows
  OzProductArgs ga{};
  ga.Asl = w.Asl;
  ga.Bsl = w.Xsl;
  ga.eA = w.eA;
  ga.eB = w.eX;
  ga.R = w.R;
  ga.M = ga.Nc = ga.K = N;
  ga.status = w.status;
  ga.weak = w.weak;
  const int* act = nullptr;
  const dim3 gref((unsigned)(N / 128), (unsigned)(N / 128), (unsigned)batch);
  if (w.weak) {
    cudaMemsetAsync(w.weak, 0, (size_t)batch * sizeof(int), st);
    cudaMemsetAsync(w.rmax, 0, (size_t)batch * sizeof(unsigned), st);
  }
  // X0: FP32 Gauss-Jordan
  {
    gw::TimedLaunch tl_("k_to_f32", st);
    k_to_f32<<<g1, 256, 0, st>>>(mats, w.X32, tot, NN, nullptr);
  }
  {
    gw::TimedLaunch tl_("k_gj_inverse_f32", st);
    if (N == 128) k_gj_inverse_f32<128><<<batch, 512, gj32_smem(N), st>>>(w.X32, Na, NN, w.status, w.weak);
    else if (N == 256) k_gj_inverse_f32<256><<<batch, 512, gj32_smem(N), st>>>(w.X32, Na, NN, w.status, w.weak);
    else k_gj_inverse_f32<384><<<batch, 512, gj32_smem(N), st>>>(w.X32, Na, NN, w.status, w.weak);
  }
  // digits of A (kept for both residuals)
  {
    gw::TimedLaunch tl_("k_row_exponent", st);
    k_row_exponent<<<(unsigned)((batch * (long long)N + 7) / 8), 256, 0, st>>>(mats, w.eA, N, batch);
  }
  {
    gw::TimedLaunch tl_("k_slice_A", st);
    if (fine) k_slice_A<kWFine><<<g8, 256, 0, st>>>(mats, w.eA, w.Asl, N, tot);
    else k_slice_A<kWSA><<<g8, 256, 0, st>>>(mats, w.eA, w.Asl, N, tot);
  }
  // R0 = I - A X0 (FP32), lo = X0 R0: X1 = X0 + lo
  {
    gw::TimedLaunch tl_("k_col_exponent", st);
    k_col_exponent<<<gcol, kCE, 0, st>>>(w.X32, nullptr, w.eX, N);
  }
  {
    gw::TimedLaunch tl_("k_slice_X", st);
    k_slice_X<kWSX0><<<g8, 256, 0, st>>>(w.X32, nullptr, w.eX, w.Xsl, N, tot);
  }
  {
    gw::TimedLaunch tl_("k_ozaki_residual<first>", st);
    if (fine) k_oz_product<kWSX0, kWL0, true, false, kWFine><<<gres, kPT, w_residual_smem(kWSX0, kWL0), st>>>(ga);
    else k_oz_product<kWSX0, kWL0, true, false, kWSA><<<gres, kPT, w_residual_smem(kWSX0, kWL0), st>>>(ga);
  }
  {
    gw::TimedLaunch tl_("k_split3_rows", st);
    k_split3_rows<<<g8, 256, 0, st>>>(w.X32, w.PX, N, tot, act);
  }
  {
    gw::TimedLaunch tl_("k_split3_cols", st);
    k_split3_cols<<<g8, 256, 0, st>>>(w.R, w.Xsl, N, tot, act);  // the X digits are no longer needed
  }
  {
    gw::TimedLaunch tl_("k_refine_tc<first>", st);
    k_refine_tc<0><<<gref, kPT, w_refine_smem(), st>>>(w.PX, w.Xsl, w.X32, w.lo, nullptr, N, w.status, act);
  }
  // R1 = I - A X1 (FP32), X2 = X1 + X0 R1 in FP64, written over A
  {
    gw::TimedLaunch tl_("k_col_exponent", st);
    k_col_exponent<<<gcol, kCE, 0, st>>>(w.X32, w.lo, w.eX, N);
  }
  {
    gw::TimedLaunch tl_("k_slice_X", st);
    k_slice_X<kWSX1><<<g8, 256, 0, st>>>(w.X32, w.lo, w.eX, w.Xsl, N, tot);
  }
  {
    gw::TimedLaunch tl_("k_ozaki_residual<second>", st);
    ga.rmax = w.rmax;
    if (fine) k_oz_product<kWSX1, kWLmax, true, true, kWFine><<<gres, kPT, w_residual_smem(kWSX1, kWLmax), st>>>(ga);
    else k_oz_product<kWSX1, kWLmax, true, true, kWSA><<<gres, kPT, w_residual_smem(kWSX1, kWLmax), st>>>(ga);
  }
  {
    gw::TimedLaunch tl_("k_split3_cols", st);
    k_split3_cols<<<g8, 256, 0, st>>>(w.R, w.Xsl, N, tot, act);
  }
  {
    gw::TimedLaunch tl_("k_refine_tc<final>", st);
    k_refine_tc<1><<<gref, kPT, w_refine_smem(), st>>>(w.PX, w.Xsl, w.X32, w.lo, mats, N, w.status, act);
  }
  // the second residual has to be small before its successor is taken modulo 2^64
  if (fine) {
    gw::TimedLaunch tl_("k_mark", st);
    k_mark<<<(unsigned)((batch + 255) / 256), 256, 0, st>>>(w.rmax, w.weak, batch, 0x1p-8f, 0);
  }
  // X <- X + X (I - A X) again, the left factor now the current X rounded to FP32 (the
  // correction is needed to 2^-24 of itself only): with X0 there the error would shrink
  // by |I - A X0| per step, with X by about kappa 2^-24 |I - A X|.  With nine digits the
  // residual is good to 2^-59 of |A||X|, so the corrected X is that of FP64 rounding; the
  // fourth refinement then takes only the matrices whose third residual was above 2^-38.
  for (int r = 3; r <= refinements; ++r) {
    {
      gw::TimedLaunch tl_("k_to_f32", st);
      k_to_f32<<<g1, 256, 0, st>>>(mats, w.X32, tot, NN, act);
    }
    {
      gw::TimedLaunch tl_("k_split3_rows", st);
      k_split3_rows<<<g8, 256, 0, st>>>(w.X32, w.PX, N, tot, act);
    }
    {
      gw::TimedLaunch tl_("k_panel_col_exp", st);
      k_panel_col_exp<<<gcol, kCE, 0, st>>>(mats, NN, N, N, N, w.eX, act);
    }
    {
      gw::TimedLaunch tl_("k_slice_panel_B", st);
      if (fine) k_slice_panel_B<kWFine><<<g8, 256, 0, st>>>(mats, NN, N, w.eX, w.Xsl, N, N, t8, act);
      else k_slice_panel_B<kWSX1><<<g8, 256, 0, st>>>(mats, NN, N, w.eX, w.Xsl, N, N, t8, act);
    }
    {
      gw::TimedLaunch tl_("k_ozaki_residual<third>", st);
      ga.rmax = w.rmax;
      ga.act = act;
      if (fine) {
        const dim3 gf((unsigned)(N / w_tn(kWFine - 1)), gres.y, gres.z);
        k_oz_product<kWFine, kWFine - 1, true, false, kWFine>
            <<<gf, kPT, w_residual_smem(kWFine, kWFine - 1), st>>>(ga);
      } else {
        k_oz_product<kWSX1, kWLmax, true, false, kWSA><<<gres, kPT, w_residual_smem(kWSX1, kWLmax), st>>>(ga);
      }
    }
    {
      gw::TimedLaunch tl_("k_split3_cols", st);
      k_split3_cols<<<g8, 256, 0, st>>>(w.R, w.Xsl, N, tot, act);
    }
    {
      gw::TimedLaunch tl_("k_refine_tc<add>", st);
      k_refine_tc<2><<<gref, kPT, w_refine_smem(), st>>>(w.PX, w.Xsl, w.X32, w.lo, mats, N, w.status, act);
    }
    if (fine) {
      gw::TimedLaunch tl_("k_mark", st);
      const bool last = r == refinements;
      k_mark<<<(unsigned)((batch + 255) / 256), 256, 0, st>>>(w.rmax, last ? w.weak : w.act, batch,
                                                               last ? 0x1p-30f : 0x1p-38f, last ? 0 : 1);
      act = w.act;
    }
  }
  if (fine) {
    // what is left: by FP64 elimination, from A's digits
    {
      gw::TimedLaunch tl_("k_unslice_A", st);
      k_unslice_A<<<dim3(16, (unsigned)batch), 256, 0, st>>>(w.Asl, w.eA, w.weak, mats, N);
    }
    gj_batch_only(mats, w.perm, batch, N, w.status, w.weak, st);
  }
}


// ---- Block Gauss-Jordan for N_PB beyond kWNmax --------------------------------------
//
// The inverse of an N x N matrix with N = nb bs (bs <= kWNmax) by Gauss-Jordan over
// blocks of bs rows and columns, without pivoting across blocks (the matrices of the W
// solve, v(q) and v(q)^-1 - P(q, i nu), are Hermitian positive definite, so every pivot
// block is too).  Pivot step k, with D = A_kk^-1 (the tensor-core inverse of bs x bs):
//   Rp = D A_k,:  (its block k replaced by I + D),
//   A_i,: -= A_ik Rp for every row block i != k   (so A_ik becomes -A_ik D),
//   A_k,: = Rp with block k = D.
// Every product has K = bs <= kWNmax terms, so it runs as the residual does: exact BF16
// digits of the two panels (per-row and per-column power-of-two scales), the level sums
// exact in FP32 tensor-memory accumulators, one exact 64-bit sum rounded once to FP64.

// Scale exponent of each row of an M x K panel (rows ld apart, matrices ms apart): one
// warp per row.
__global__ void k_panel_row_exp(const double2* __restrict__ A, long long ms, int ld, int M, int K, int batch,
                                int* __restrict__ e) {
  const int warps = blockDim.x >> 5;
  const long long row = (long long)blockIdx.x * warps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= (long long)batch * M) return;
  const long long b = row / M, i = row % M;
  const double2* a = A + b * ms + i * ld;
  int m = 0;
  for (int k = lane; k < K; k += 32) m = max(m, max(exp_field(a[k].x), exp_field(a[k].y)));
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) e[row] = m > 0 ? m - 1022 : 0;
}

// Scale exponent of each column of a K x Nc panel: blocks as in k_col_exponent.
__global__ void __launch_bounds__(kCE) k_panel_col_exp(const double2* __restrict__ B, long long ms, int ld, int K, int Nc,
                                                       int* __restrict__ e, const int* __restrict__ act) {
  const int b = blockIdx.y, j = blockIdx.x * 32 + (threadIdx.x & 31);
  if (act && !act[b]) return;
  const double2* c = B + (long long)b * ms + j;
  int m = 0;
  if (j < Nc)
#pragma unroll 4
    for (int k = threadIdx.x >> 5; k < K; k += 8) {
      const double2 z = c[(long long)k * ld];
      m = max(m, max(exp_field(z.x), exp_field(z.y)));
    }
  m = col_max(m);
  if (threadIdx.x < 32 && j < Nc) e[(long long)b * Nc + j] = m > 0 ? m - 1022 : 0;
}

// A-operand digits of an M x K panel, chunks as k_slice_A: one per (matrix, 128-row
// block, 16-wide K step) with the kWSA digits of Re, then of Im.
__global__ void k_slice_panel_A(const double2* __restrict__ A, long long ms, int ld, const int* __restrict__ eA,
                                uint16_t* __restrict__ Asl, int M, int K, long long n_thr) {
  const int NKS = K / 16, NIB = M / 128;
  for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < n_thr; x += (long long)gridDim.x * blockDim.x) {
    const int lane = (int)(x & 31);
    long long w = x >> 5;  // (b, ib, ks, row group pair)
    const int gp = (int)(w % 8); w /= 8;
    const int ks = (int)(w % NKS); w /= NKS;
    const int ib = (int)(w % NIB);
    const long long b = w / NIB;
    const int h = (lane >> 3) & 1;
    const int il = (lane & 7) + 8 * ((lane >> 4) + 2 * gp);
    const int i = ib * 128 + il;
    const int k0 = ks * 16 + 8 * h;
    const int e = eA[b * M + i];
    const double2* src = A + b * ms + (long long)i * ld + k0;
    long long mr[8], mi[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double2 z = src[u];
      mr[u] = fixed56(z.x, e);
      mi[u] = fixed56(z.y, e);
    }
    uint16_t* chunk = Asl + ((b * NIB + ib) * NKS + ks) * (long long)(kWAChunk / 2);
    const uint32_t off = kmajor_offset(128, il, 8 * h) / 2;
#pragma unroll
    for (int s = 0; s < kWSA; ++s) {
      uint32_t pr[4], pi[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t r0 = digit_bf16(next_digit(mr[2 * u], s), s), r1 = digit_bf16(next_digit(mr[2 * u + 1], s), s);
        const uint32_t i0 = digit_bf16(next_digit(mi[2 * u], s), s), i1 = digit_bf16(next_digit(mi[2 * u + 1], s), s);
        pr[u] = r0 | (r1 << 16);
        pi[u] = i0 | (i1 << 16);
      }
      *reinterpret_cast<uint4*>(chunk + (0 * kWSA + s) * (128 * 16) + off) = make_uint4(pr[0], pr[1], pr[2], pr[3]);
      *reinterpret_cast<uint4*>(chunk + (1 * kWSA + s) * (128 * 16) + off) = make_uint4(pi[0], pi[1], pi[2], pi[3]);
    }
  }
}

// B-operand digits of a K x Nc panel (FP64), chunks as k_slice_X: one per (matrix, column
// block, 16-wide K step) with the ND digits of Re, then of Im (blocks of kWTN columns, or of
// the narrower ones of nine digits).
template <int ND>
__global__ void k_slice_panel_B(const double2* __restrict__ B, long long ms, int ld, const int* __restrict__ eB,
                                uint16_t* __restrict__ Bsl, int K, int Nc, long long n_thr,
                                const int* __restrict__ act) {
  constexpr int TN = w_tn(ND - 1), JG = TN / 16;
  const int NKS = K / 16, NJB = Nc / TN;
  for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < n_thr; x += (long long)gridDim.x * blockDim.x) {
    const int lane = (int)(x & 31);
    long long w = x >> 5;  // (b, jb, ks, column group)
    const int jg = (int)(w % JG); w /= JG;
    const int ks = (int)(w % NKS); w /= NKS;
    const int jb = (int)(w % NJB);
    const long long b = w / NJB;
    if (act && !act[b]) continue;
    const int h = (lane >> 3) & 1;
    const int jl = (lane & 7) + 8 * ((lane >> 4) + 2 * jg);
    const int j = jb * TN + jl;
    const int k0 = ks * 16 + 8 * h;
    const int e = eB[b * Nc + j];
    const double2* src = B + b * ms + (long long)k0 * ld + j;
    long long mr[8], mi[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double2 z = src[(long long)u * ld];
      mr[u] = fixed_nd<ND>(z.x, e);
      mi[u] = fixed_nd<ND>(z.y, e);
    }
    uint16_t* chunk = Bsl + ((b * NJB + jb) * NKS + ks) * (long long)(wx_chunk(ND, TN) / 2);
    const uint32_t off = kmajor_offset(TN, jl, 8 * h) / 2;
#pragma unroll
    for (int t = 0; t < ND; ++t) {
      uint32_t pr[4], pi[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t r0 = digit_bf16(digit_nd<ND>(mr[2 * u], t), t), r1 = digit_bf16(digit_nd<ND>(mr[2 * u + 1], t), t);
        const uint32_t i0 = digit_bf16(digit_nd<ND>(mi[2 * u], t), t), i1 = digit_bf16(digit_nd<ND>(mi[2 * u + 1], t), t);
        pr[u] = r0 | (r1 << 16);
        pi[u] = i0 | (i1 << 16);
      }
      *reinterpret_cast<uint4*>(chunk + (0 * ND + t) * (TN * 16) + off) = make_uint4(pr[0], pr[1], pr[2], pr[3]);
      *reinterpret_cast<uint4*>(chunk + (1 * ND + t) * (TN * 16) + off) = make_uint4(pi[0], pi[1], pi[2], pi[3]);
    }
  }
}

// dst[b][r][c] = src[b][r][c] (+ 1 on the diagonal r == c when add_identity), r < rows,
// c < cols, for matrices of row strides sld / dld and matrix strides sms / dms.
__global__ void k_copy_panel(const double2* __restrict__ src, long long sms, int sld, double2* __restrict__ dst,
                             long long dms, int dld, int rows, int cols, int batch, int add_identity) {
  const long long per = (long long)rows * cols, n = per * batch;
  for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (long long)gridDim.x * blockDim.x) {
    const long long b = x / per, rc = x % per;
    const int r = (int)(rc / cols), c = (int)(rc % cols);
    double2 z = src[b * sms + (long long)r * sld + c];
    if (add_identity && r == c) z.x += 1.0;
    dst[b * dms + (long long)r * dld + c] = z;
  }
}


namespace {

unsigned grid_for(long long n_thr) {
  const long long g = (n_thr + 255) / 256;
  return (unsigned)(g < 65535LL * 8 ? (g > 0 ? g : 1) : 65535LL * 8);
}

// C (M x Nc, rows ldc apart, matrices c_ms apart) = / -= A B for the panels A (M x K at
// A, rows lda apart) and B (K x Nc at B, rows ldb apart), every matrix of the batch.
void panel_gemm(const WblkBuffers& w, const double2* A, long long a_ms, int lda, const double2* B, long long b_ms,
                int ldb, double2* C, long long c_ms, int ldc, int M, int Nc, int K, int batch, int skip0, int skip1,
                int accumulate, cudaStream_t st) {
  {
    gw::TimedLaunch tl_("k_panel_row_exp", st);
    k_panel_row_exp<<<(unsigned)((batch * (long long)M + 7) / 8), 256, 0, st>>>(A, a_ms, lda, M, K, batch, w.eA);
  }
  {
    gw::TimedLaunch tl_("k_slice_panel_A", st);
    k_slice_panel_A<<<grid_for((long long)batch * M * K / 8), 256, 0, st>>>(A, a_ms, lda, w.eA, w.Asl, M, K,
                                                                             (long long)batch * M * K / 8);
  }
  {
    gw::TimedLaunch tl_("k_panel_col_exp", st);
    k_panel_col_exp<<<dim3((unsigned)((Nc + 31) / 32), (unsigned)batch), kCE, 0, st>>>(B, b_ms, ldb, K, Nc, w.eB, nullptr);
  }
  {
    gw::TimedLaunch tl_("k_slice_panel_B", st);
    k_slice_panel_B<kWSX1><<<grid_for((long long)batch * K * Nc / 8), 256, 0, st>>>(
        B, b_ms, ldb, w.eB, w.Bsl, K, Nc, (long long)batch * K * Nc / 8, nullptr);
  }
  OzProductArgs g{};
  g.Asl = w.Asl;
  g.Bsl = w.Bsl;
  g.eA = w.eA;
  g.eB = w.eB;
  g.C = C;
  g.c_ms = c_ms;
  g.ldc = ldc;
  g.M = M;
  g.Nc = Nc;
  g.K = K;
  g.skip0 = skip0;
  g.skip1 = skip1;
  g.accumulate = accumulate;
  g.status = w.inner.status;
  {
    gw::TimedLaunch tl_("k_oz_panel_gemm", st);
    k_oz_product<kWSX1, kWLmax, false, false, kWSA><<<dim3((unsigned)(Nc / kWTN), (unsigned)(2 * (M / 128)), (unsigned)batch), kPT,
                                         w_residual_smem(kWSX1, kWLmax), st>>>(g);
  }
}

void copy_panel(const double2* src, long long sms, int sld, double2* dst, long long dms, int dld, int rows, int cols,
                int batch, int add_identity, cudaStream_t st) {
  gw::TimedLaunch tl_("k_copy_panel", st);
  k_copy_panel<<<grid_for((long long)batch * rows * cols), 256, 0, st>>>(src, sms, sld, dst, dms, dld, rows, cols,
                                                                          batch, add_identity);
}

}  // namespace

int wblk_block_size(int N) {
  if (N <= kWNmax || N % 128 != 0) return 0;
  for (int bs = kWblkMaxK; bs >= 128; bs -= 128)
    if (N % bs == 0) return bs;
  return 0;
}

cudaError_t wblk_setup() {
  cudaError_t e = wtc_setup();
  if (e == cudaSuccess) e = raise_smem_limit(k_oz_product<kWSX1, kWLmax, false, false, kWSA>, w_residual_smem(kWSX1, kWLmax));
  return e;
}

void wblk_inverse(const WblkBuffers& w, double2* mats, int batch, int N, int bs, cudaStream_t st) {
  const long long NN = (long long)N * N, BB = (long long)bs * bs, BN = (long long)bs * N;
  for (int k = 0; k < N / bs; ++k) {
    const int r0 = k * bs;
    // D = A_kk^-1
    copy_panel(mats + (long long)r0 * N + r0, NN, N, w.D, BB, bs, bs, bs, batch, 0, st);
    wtc_inverse(w.inner, w.D, batch, bs, st, kWblkRefinements);
    // Rp = D A_k,: with block k = I + D
    panel_gemm(w, w.D, BB, bs, mats + (long long)r0 * N, NN, N, w.Rp, BN, N, bs, N, bs, batch, 0, 0, 0, st);
    copy_panel(w.D, BB, bs, w.Rp + r0, BN, N, bs, bs, batch, 1, st);
    // A_i,: -= A_ik Rp for the other row blocks (the column panel is sliced before any write)
    panel_gemm(w, mats + r0, NN, N, w.Rp, BN, N, mats, NN, N, N, N, bs, batch, r0 / 128, (r0 + bs) / 128, 1, st);
    // A_k,: = Rp with block k = D
    copy_panel(w.Rp, BN, N, mats + (long long)r0 * N, NN, N, bs, N, batch, 0, st);
    copy_panel(w.D, BB, bs, mats + (long long)r0 * N + r0, NN, N, bs, bs, batch, 0, st);
  }
}

}  // namespace gw
