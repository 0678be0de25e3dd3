// FP64 P (Eq. P_MM) and Sigma (Eq. S_MM) for product coefficients symmetric in (L, L''), as
// contractions over the symmetric orbital pairs p = (L <= L''), n (n + 1) / 2 of them:
//
//   P[K][K']  = -s sum_pq C^a[K][p] M[p][q] C^b[K'][q],
//     M[p][q] = G(tau) conj(G(beta - tau)) summed over the orderings of both pairs,
//   D[p][q]   = sum_KK' C^a[K][p] W~[K][K'] C^b[K'][q],   Sigma[L][L'] = -sum_{L'' L'''}
//               D[(L, L'')][(L', L''')] G[L''][L'''].
//
// In FP64 arithmetic that leaves n_a^2 n_b^2 complex multiply-adds per unit (entry, node)
// beside two real-times-complex products, which run as exact base-2^7 digit products on
// tcgen05 (oz.h): at n = 9, K = 48 the FP64 pipe (two multiply-adds per clock and SM) does
// 26 thousand instead of 210 thousand for P and 280 thousand for Sigma, and what is left on it
// takes as long as the tensor-core chain.
//
//   k_polarizability_pairs   M in FP64, cut into digits: rows (c, p), reduction q
//   k_slice_w_units          W~ cut into digits: rows (c, K), reduction K'
//   k_chain                  first product, cut into digits without leaving the SM, second product
//   k_sigma_pairs            the last sum of Sigma in FP64
//
// A unit's 128 operand rows are two halves of 64: real, then imaginary parts.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <vector>

#include "chain.h"
#include "kernels.h"
#include "ktimer.h"
#include "ozdigits.h"
#include "smem_limit.h"

namespace gw {

namespace {

constexpr uint64_t kChWaitNs = 500ull * 1000ull * 1000ull;
constexpr uint32_t kChStep = kOzDigits * kTfPlane;  // 32 KB: digits of 128 rows, one 16-wide K step

__host__ __device__ constexpr uint32_t ch_bstep(int NT) { return (uint32_t)kOzDigits * NT * 32; }

// Digits of 8 values of one row to global memory: K half h of step ks of unit base A.
__device__ __forceinline__ void ch_store_row(unsigned char* A, int r, int k8, const long long* m) {
  tf_cut8(m, A + (k8 >> 1) * kChStep + kmajor_offset(128, r, 8 * (k8 & 1)));
}

// ---------------------------------------------------------------------------------------
// M of one unit (entry blockIdx.x, node s0 + blockIdx.y) and its digits.  Bound by the FP64
// pipe: four multiply-adds per ordering.  The rows' scales need all of a row, so M goes
// through shared memory once.  9024 units of n = 9: 0.48 ms, 0.41 of it FP64 issue; stages X and Y of the
// other path took 3.13 ms.
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_polarizability_pairs(const DevEntry* __restrict__ ent,
                                                              const int* __restrict__ species,
                                                              const unsigned char* __restrict__ pairs,
                                                              const double2* __restrict__ G, int n_tau, int s0, int KS,
                                                              uint16_t* __restrict__ Adig, int* __restrict__ eA) {
  extern __shared__ double2 smp[];
  __shared__ unsigned char pa[2][kChainMax], pb[2][kChainMax];
  __shared__ int e_s[128];
  const DevEntry E = ent[blockIdx.x];
  const int na = E.na, nb = E.nb, np = na * (na + 1) / 2, nq = nb * (nb + 1) / 2, ldq = nq | 1;
  const long long unit = (long long)blockIdx.x * gridDim.y + blockIdx.y;
  const int it = s0 + blockIdx.y, im = n_tau - 1 - it;
  double2* g1 = smp;              // [na][nb] G(tau)
  double2* g2 = g1 + na * nb;     // [na][nb] conj(G(beta - tau))
  double2* M = g2 + na * nb;      // [np][ldq]
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const double2* Gin = G + E.off_orb * n_tau;
  for (int x = t; x < na * nb; x += 256) {
    g1[x] = Gin[(long long)it * na * nb + x];
    const double2 z = Gin[(long long)im * na * nb + x];
    g2[x] = make_double2(z.x, dneg(z.y));
  }
  if (t < 2 * kChainMax) {
    pa[t / kChainMax][t % kChainMax] = pairs[species[E.a] * 2 * kChainMax + t];
    pb[t / kChainMax][t % kChainMax] = pairs[species[E.b] * 2 * kChainMax + t];
  }
  if (t < 128) e_s[t] = 0;
  __syncthreads();
  // the diagonal pairs come first, so a warp mostly takes one number of orderings
  for (int x = t; x < np * nq; x += 256) {
    const int p = x / nq, q = x - p * nq;
    const int L = pa[0][p] * nb, L2 = pa[1][p] * nb, L1 = pb[0][q], L3 = pb[1][q];
    auto mul = [&](int i, int j, double2 acc) {
      const double2 a = g1[i], b = g2[j];
      return make_double2(fma(a.x, b.x, fma(-a.y, b.y, acc.x)), fma(a.x, b.y, fma(a.y, b.x, acc.y)));
    };
    double2 acc = mul(L + L1, L2 + L3, make_double2(0.0, 0.0));
    if (L1 != L3) acc = mul(L + L3, L2 + L1, acc);
    if (L != L2) {
      acc = mul(L2 + L1, L + L3, acc);
      if (L1 != L3) acc = mul(L2 + L3, L + L1, acc);
    }
    M[p * ldq + q] = acc;
  }
  __syncthreads();
  for (int p = wid; p < np; p += 8) {
    int mr = 0, mi = 0;
    for (int q = lane; q < nq; q += 32) {
      const double2 z = M[p * ldq + q];
      mr = max(mr, exp_field(z.x));
      mi = max(mi, exp_field(z.y));
    }
    mr = __reduce_max_sync(0xffffffffu, mr);
    mi = __reduce_max_sync(0xffffffffu, mi);
    if (lane == 0) {
      e_s[p] = tf_row_scale(mr);
      e_s[64 + p] = tf_row_scale(mi);
    }
  }
  __syncthreads();
  if (t < 128) eA[unit * 128 + t] = e_s[t];
  unsigned char* A = reinterpret_cast<unsigned char*>(Adig) + unit * KS * kChStep;
  // 8 lanes on the rows of a core matrix, both K halves beside them: 512 contiguous bytes per warp
  for (int x = t; x < 64 * 2 * KS; x += 256) {
    const int p = (x & 7) | ((x >> 4) & 7) << 3, k8 = ((x >> 3) & 1) | (x >> 7) << 1;
    long long R[8], I[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int q = 8 * k8 + u;
      const double2 z = p < np && q < nq ? M[p * ldq + q] : make_double2(0.0, 0.0);
      R[u] = fixed56(z.x, e_s[p]);
      I[u] = fixed56(z.y, e_s[64 + p]);
    }
    ch_store_row(A, p, k8, R);
    ch_store_row(A, 64 + p, k8, I);
  }
}

// W~ (or v) of one unit cut into digits: rows (c, K), reduction K'.
__global__ void __launch_bounds__(256) k_slice_w_units(const DevEntry* __restrict__ ent, const double2* __restrict__ W,
                                                       int n_slices, int s0, int KS, uint16_t* __restrict__ Adig,
                                                       int* __restrict__ eA) {
  __shared__ int e_s[128];
  const DevEntry E = ent[blockIdx.x];
  const int Ka = E.Ka, Kb = E.Kb;
  const long long unit = (long long)blockIdx.x * gridDim.y + blockIdx.y;
  const double2* w = W + E.off_pb * n_slices + (long long)(s0 + blockIdx.y) * Ka * Kb;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  if (t < 128) e_s[t] = 0;
  __syncthreads();
  for (int K = wid; K < Ka; K += 8) {
    int mr = 0, mi = 0;
    for (int k = lane; k < Kb; k += 32) {
      const double2 z = w[(long long)K * Kb + k];
      mr = max(mr, exp_field(z.x));
      mi = max(mi, exp_field(z.y));
    }
    mr = __reduce_max_sync(0xffffffffu, mr);
    mi = __reduce_max_sync(0xffffffffu, mi);
    if (lane == 0) {
      e_s[K] = tf_row_scale(mr);
      e_s[64 + K] = tf_row_scale(mi);
    }
  }
  __syncthreads();
  if (t < 128) eA[unit * 128 + t] = e_s[t];
  unsigned char* A = reinterpret_cast<unsigned char*>(Adig) + unit * KS * kChStep;
  for (int x = t; x < 64 * 2 * KS; x += 256) {
    const int K = (x & 7) | ((x >> 4) & 7) << 3, k8 = ((x >> 3) & 1) | (x >> 7) << 1;
    long long R[8], I[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = 8 * k8 + u;
      const double2 z = K < Ka && k < Kb ? w[(long long)K * Kb + k] : make_double2(0.0, 0.0);
      R[u] = fixed56(z.x, e_s[K]);
      I[u] = fixed56(z.y, e_s[64 + K]);
    }
    ch_store_row(A, K, k8, R);
    ch_store_row(A, 64 + K, k8, I);
  }
}

// ---------------------------------------------------------------------------------------
// The two products of a unit.  Rows of the first operand: (c, r) with r < 64 the reduction
// index of the second product; its columns n become the rows (c, n) of the second operand.
// The first product's exact 64-bit sums are cut into digits again at one power-of-two scale
// per row (c, n) and written as an M-major operand (8 consecutive n per 16 bytes: the lane
// holds one r and consecutive n), so they neither leave the SM nor round in between.
// Persistent, one block per SM; each warp has 32 rows x kW columns, 8 of them where the
// registers allow that many warps: the read-outs and cuts are integer work, about as much as
// the products take, and three warps per scheduler (16 columns each) left half its issue
// slots idle.  The digits of the next unit come in by bulk copies while this one's second
// product is read out.  P goes out through shared memory, so that a store is 16 bytes of 32
// consecutive K' (from the accumulators' lanes it would be the real or the imaginary halves).
// 9024 units of n = 9, K = 48: 0.69 ms for P (with 16 columns per warp and halves stored from
// the lanes 0.03 ms more), 18424 units of Sigma 1.22 ms (0.18 more).  Prefetching the next unit's
// digits into L2 changed nothing (0.74 ms): they are there.
// ---------------------------------------------------------------------------------------
struct ChainArgs {
  const DevEntry* ent;
  const int* species;
  int n_units, tau_eff;  // unit = entry tau_eff + slice of the pass
  int KS;
  const uint16_t* Adig;
  const int* eA;
  const uint16_t* B;     // static operands of all species: that of b in the first product, of a in the second
  const int* eB;
  int eB_min, eB_max;
  // P: out[e][s0 + slice][n2 .. ] = -s value at row K = column of the second product, K' = its row
  double2* P;
  int n_tau, s0, ms_shift;
  // Sigma: D[unit][n2][(c, n1)]
  double* D;
  int ld_d;
  int* status;
};

__host__ __device__ constexpr int ch_w(int NT) { return NT <= 48 ? 8 : 16; }          // columns per warp
__host__ __device__ constexpr int ch_threads(int NT) { return 128 * (NT / ch_w(NT)); }
// P staging per column group of four warps: 8 columns x 64 rows, real and imaginary planes
__host__ __device__ constexpr uint32_t ch_stage(int NT) { return (uint32_t)(NT / ch_w(NT)) * 8 * 64 * 16; }

// The 64-bit sums (units of 2^-56 of the scale, below 64 of it: 64 terms) of W columns of this
// thread's row: eight level accumulators NT columns apart at taddr, each an integer below 2^22
// of its unit.
template <int W>
__device__ __forceinline__ void ch_sums(uint32_t taddr, uint32_t NT, long long* S) {
#pragma unroll
  for (int c0 = 0; c0 < W; c0 += 8) {
#pragma unroll
    for (int j = 0; j < 8; ++j) S[c0 + j] = 0;
#pragma unroll
    for (int l = 0; l < 8; l += 4) {
      float v[32];
      tmem_ld8x4(taddr + (uint32_t)c0 + (uint32_t)l * NT, NT, v);
#pragma unroll
      for (int q = 0; q < 4; q += 2) {
        const float s0 = __int_as_float((127 + 7 * (l + q)) << 23), s1 = __int_as_float((127 + 7 * (l + q + 1)) << 23);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int P = tf_pair_int<false>(v[8 * q + j], s0, v[8 * q + 8 + j], s1);
          if (l + q < 6) S[c0 + j] += (long long)P << (42 - 7 * (l + q + 1));
          else S[c0 + j] += (long long)((P + 64) >> 7);  // level 7: rounded at 2^-56
        }
      }
    }
  }
}

template <int NT, bool SIGMA>
__global__ void __launch_bounds__(ch_threads(NT), 1) k_chain(const __grid_constant__ ChainArgs g) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint32_t tmem_base;
  __shared__ __align__(8) uint64_t full, b_full, done;
  __shared__ int row_e[128];
  __shared__ int eB1[NT], eB2[NT];
  const int KS = g.KS;
  const uint32_t BB = KS * ch_bstep(NT);
  unsigned char* A = sm;
  unsigned char* B1 = sm + KS * kChStep;
  unsigned char* B2 = B1 + BB;
  constexpr int W = ch_w(NT);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row = 32 * (warp & 3) + lane, c = row >> 6, r = row & 63, n0 = W * (warp >> 2);
  if (warp == 0) {
    tmem_alloc(&tmem_base, 512);
    tmem_relinquish();
  }
  if (tid == 0) {
    mbar_init(&full, 1);
    mbar_init(&b_full, 1);
    mbar_init(&done, 1);
    fence_mbar_init();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tm = tmem_base;
  const uint32_t t_addr = tm + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)n0;
  auto load_a = [&](int u) {
    mbar_arrive_expect_tx(&full, KS * kChStep);
    const unsigned char* src = reinterpret_cast<const unsigned char*>(g.Adig) + (long long)u * KS * kChStep;
    for (int ks = 0; ks < KS; ++ks) bulk_g2s(A + ks * kChStep, src + (long long)ks * kChStep, kChStep, &full);
  };
  bool ok = true;
  int cur1 = -1, cur2 = -1, b_loads = 0;
  uint32_t ph_done = 0, ph_full = 0;
  if (tid == 0 && (int)blockIdx.x < g.n_units) load_a(blockIdx.x);
  for (int u = blockIdx.x; u < g.n_units; u += gridDim.x) {
    const int e = u / g.tau_eff, sl = u - e * g.tau_eff;
    const DevEntry E = g.ent[e];
    const int s1 = g.species[E.b], s2 = g.species[E.a];
    const int ea = g.eA[(long long)u * 128 + row];  // row scale exponent
    if (s1 != cur1 || s2 != cur2) {  // the static operands of another species pair
      if (tid == 0) {
        mbar_arrive_expect_tx(&b_full, 2 * BB);
        bulk_g2s(B1, reinterpret_cast<const unsigned char*>(g.B) + (size_t)s1 * BB, BB, &b_full);
        bulk_g2s(B2, reinterpret_cast<const unsigned char*>(g.B) + (size_t)s2 * BB, BB, &b_full);
      }
      for (int j = tid; j < NT; j += ch_threads(NT)) {
        eB1[j] = g.eB[s1 * NT + j];
        eB2[j] = g.eB[s2 * NT + j];
      }
      const bool got = mbar_wait(&b_full, (uint32_t)b_loads & 1u, kChWaitNs, g.status);
      ok = __syncthreads_and(got ? 1 : 0) != 0;
      if (!ok) break;
      ++b_loads;
      cur1 = s1;
      cur2 = s2;
    }
    if (tid < 128) row_e[tid] = -100000;
    if (tid == 0) {
      ok = mbar_wait(&full, ph_full, kChWaitNs, g.status);
      fence_after_sync();
      if (ok) {
        const uint32_t a0 = smem_u32(A), b0 = smem_u32(B1);
        for (int ks = 0; ks < KS; ++ks)
          tf_issue_step<NT>(tm, smem_desc(a0 + ks * kChStep, 128, 256), smem_desc(b0 + ks * ch_bstep(NT), 128, 256), ks == 0);
      } else {
        atomicExch(g.status, 2);
      }
      mma_commit(&done);
    }
    ph_full ^= 1u;
    __syncwarp();
    ok = mbar_wait(&done, ph_done, kChWaitNs, g.status) && ok;
    ph_done ^= 1u;
    ok = __syncthreads_and(ok ? 1 : 0) != 0;
    fence_after_sync();
    if (!ok) break;
    long long S[W];
    ch_sums<W>(t_addr, NT, S);
    // the scale of each row (c, n) of the second operand: the largest value over r
    int mine = -100000;
    const int none = ea > kOzNaN / 2 ? ea : -100000;  // of a zero sum
#pragma unroll
    for (int j = 0; j < W; ++j) {
      const long long a = S[j] ^ (S[j] >> 63);  // |S| <= a + 1
      const int ex = S[j] ? 64 - __clzll(a) + ea + eB1[n0 + j] - 56 : none;
      const int m = __reduce_max_sync(0xffffffffu, ex);
      if (lane == j) mine = m;
    }
    if (lane < W) atomicMax(&row_e[64 * c + n0 + lane], mine);
    fence_before_sync();
    __syncthreads();
    if (r < 16 * KS) {
#pragma unroll
      for (int h = 0; h < W / 8; ++h) {
        long long M[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int em = row_e[64 * c + n0 + 8 * h + j];
          M[j] = em > -100000 ? shift_round(S[8 * h + j], ea + eB1[n0 + 8 * h + j] - em) : 0ll;
        }
        // M-major core matrices: 8 reduction indices of 16 bytes, 8 rows (c, n) in each
        unsigned char* a = A + (r >> 4) * kChStep + ((64 * c + n0) / 8 + h) * 256 + ((r >> 3) & 1) * 128 + (r & 7) * 16;
        tf_cut8(M, a);
      }
    }
    const int er = row_e[row];  // of this thread's row of the second product
    fence_smem_to_async();
    fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      fence_after_sync();
      const uint32_t a0 = smem_u32(A), b0 = smem_u32(B2);
      for (int ks = 0; ks < KS; ++ks)
        tf_issue_step<NT>(tm, smem_desc(a0 + ks * kChStep, 128, 256), smem_desc(b0 + ks * ch_bstep(NT), 128, 256), ks == 0,
                          1u << 15);  // A is M-major
      mma_commit(&done);
    }
    __syncwarp();
    ok = mbar_wait(&done, ph_done, kChWaitNs, g.status);
    ph_done ^= 1u;
    ok = __syncthreads_and(ok ? 1 : 0) != 0;
    fence_after_sync();
    if (!ok) break;
    if (tid == 0 && u + (int)gridDim.x < g.n_units) load_a(u + gridDim.x);
    ch_sums<W>(t_addr, NT, S);
    fence_before_sync();  // ordered before the next unit's products by the barrier below
    // every result of the warp zero or a normal number (|S| < 2^62)?
    const bool normal = __all_sync(0xffffffffu, er <= -100000 || (er + g.eB_min - 56 >= -1022 && er + g.eB_max + 8 <= 1023));
    auto slow = [&](long long s, int e) { return er > -100000 ? tf_i2d_any(s, e) : 0.0; };
    if (SIGMA) {
      // lanes on consecutive doubles of one n2
      double* d = g.D + (long long)u * g.ld_d * 128 + row;
      if (normal) {
#pragma unroll
        for (int j = 0; j < W; ++j)
          if (n0 + j < g.ld_d) d[(n0 + j) * 128] = tf_i2d(S[j], er + eB2[n0 + j] - 56);
      } else {
#pragma unroll
        for (int j = 0; j < W; ++j)
          if (n0 + j < g.ld_d) d[(n0 + j) * 128] = slow(S[j], er + eB2[n0 + j] - 56);
      }
    } else {
      const int grp = warp >> 2, tg = tid & 127;
      double* stg = reinterpret_cast<double*>(B2 + BB) + grp * (8 * 64 * 2);
      const int it = g.s0 + sl, im = g.n_tau - 1 - it;
      double2* o = g.P + E.off_pb * g.n_tau + (long long)it * E.Ka * E.Kb;
      const long long moff = (long long)(im - it) * E.Ka * E.Kb;
#pragma unroll
      for (int h = 0; h < W / 8; ++h) {
        if (h > 0) asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory");
        // -s (s = 1 or 2) folded into the integer and the exponent
        if (normal) {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            stg[(2 * j + c) * 64 + r] = tf_i2d(-S[8 * h + j], er + eB2[n0 + 8 * h + j] - 56 + g.ms_shift);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            stg[(2 * j + c) * 64 + r] = slow(-S[8 * h + j], er + eB2[n0 + 8 * h + j] - 56 + g.ms_shift);
        }
        asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory");
        const int Kp = tg & 63;
#pragma unroll
        for (int j = tg >> 6; j < 8; j += 2) {
          const int K = n0 + 8 * h + j;
          if (Kp < E.Kb && K < E.Ka) {
            const double re = stg[2 * j * 64 + Kp], im_ = stg[(2 * j + 1) * 64 + Kp];
            double2* q = o + (long long)K * E.Kb + Kp;
            *q = make_double2(re, im_);
            if (moff) q[moff] = make_double2(re, dneg(im_));  // the mirrored node is the conjugate
          }
        }
      }
    }
    __syncthreads();  // row_e and the accumulators are read
  }
  if (!ok && tid == 0) {
    atomicExch(g.status, 2);
    // what was issued last ends before the memory is given back
    mbar_wait(&done, ph_done, kChWaitNs, nullptr);
    mbar_wait(&full, ph_full, kChWaitNs, nullptr);
  }
  fence_before_sync();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tm, 512);
}

// ---------------------------------------------------------------------------------------
// Sigma[L][L'] = sign sum_{L'' L'''} D[(L, L'')][(L', L''')] G[L''][L'''], one unit per block.
// Bound by the FP64 pipe: n_a^2 n_b^2 complex multiply-adds.  A thread takes one (L, L') and
// every n_seg-th L''.  18048 units of n = 9: 0.84 ms, 0.80 of it FP64 issue.
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_sigma_pairs(const DevEntry* __restrict__ ent, const int* __restrict__ species,
                                                     const unsigned char* __restrict__ pidx,
                                                     const double* __restrict__ D, int ld_d,
                                                     const double2* __restrict__ G, int g_slices, int g_fixed, int s0,
                                                     double sign, double2* __restrict__ out, int out_slices) {
  extern __shared__ double sms[];
  __shared__ unsigned char ia[256], ib[256];
  __shared__ double2 gs[256];
  const DevEntry E = ent[blockIdx.x];
  const int na = E.na, nb = E.nb, np = na * (na + 1) / 2, nq = nb * (nb + 1) / 2;
  const long long unit = (long long)blockIdx.x * gridDim.y + blockIdx.y;
  const int s = s0 + blockIdx.y;
  double2* d = reinterpret_cast<double2*>(sms);  // [np][nq]
  const double* du = D + unit * ld_d * 128;
  const int t = threadIdx.x;
  for (int x = t; x < np * nq; x += 256) {
    const int p = x / nq, q = x - p * nq;
    d[x] = make_double2(du[p * 128 + q], du[p * 128 + 64 + q]);
  }
  const double2* Gin = G + E.off_orb * g_slices + (long long)(g_fixed >= 0 ? g_fixed : s) * na * nb;
  if (t < na * nb) gs[t] = Gin[t];
  ia[t] = pidx[species[E.a] * 256 + t];
  ib[t] = pidx[species[E.b] * 256 + t];
  __syncthreads();
  const int no = na * nb, n_seg = 256 / no;  // segments of L'' (na nb <= 121)
  const int seg = t / no, o = t - seg * no;
  double2 acc = make_double2(0.0, 0.0);
  if (seg < n_seg) {
    const int L = o / nb, L1 = o - (o / nb) * nb;
    for (int L2 = seg; L2 < na; L2 += n_seg) {
      const double2* dp = d + ia[L * 16 + L2] * nq;
      for (int L3 = 0; L3 < nb; ++L3) {
        const double2 x = dp[ib[L1 * 16 + L3]], y = gs[L2 * nb + L3];
        acc = make_double2(fma(x.x, y.x, fma(-x.y, y.y, acc.x)), fma(x.x, y.y, fma(x.y, y.x, acc.y)));
      }
    }
  }
  __syncthreads();
  if (seg < n_seg) d[t] = acc;
  __syncthreads();
  if (t < no) {
    double2 a = d[t];
    for (int i = 1; i < n_seg; ++i) {
      a.x += d[t + i * no].x;
      a.y += d[t + i * no].y;
    }
    out[E.off_orb * out_slices + (long long)s * no + t] = make_double2(sign * a.x, sign * a.y);
  }
}

template <bool SIGMA>
size_t chain_smem(const ChainTable& t) {
  // more than half of the SM's shared memory: one block per SM, so that no two blocks compete
  // for the tensor memory
  return std::max((size_t)t.KS * (kChStep + 2 * ch_bstep(t.NT)) + (SIGMA ? 0 : ch_stage(t.NT)), (size_t)116 * 1024);
}

template <bool SIGMA>
cudaError_t chain_raise(const ChainTable& t) {
  switch (t.NT) {
    case 16: return raise_smem_limit(k_chain<16, SIGMA>, chain_smem<SIGMA>(t));
    case 32: return raise_smem_limit(k_chain<32, SIGMA>, chain_smem<SIGMA>(t));
    case 48: return raise_smem_limit(k_chain<48, SIGMA>, chain_smem<SIGMA>(t));
    default: return raise_smem_limit(k_chain<64, SIGMA>, chain_smem<SIGMA>(t));
  }
}
template <bool SIGMA>
void chain_launch(const ChainTable& t, const ChainArgs& a, int n_sm, cudaStream_t st) {
  TimedLaunch tl_("k_chain", st);
  const unsigned grid = (unsigned)std::min(a.n_units, n_sm);
  switch (t.NT) {
    case 16: k_chain<16, SIGMA><<<grid, ch_threads(16), chain_smem<SIGMA>(t), st>>>(a); break;
    case 32: k_chain<32, SIGMA><<<grid, ch_threads(32), chain_smem<SIGMA>(t), st>>>(a); break;
    case 48: k_chain<48, SIGMA><<<grid, ch_threads(48), chain_smem<SIGMA>(t), st>>>(a); break;
    default: k_chain<64, SIGMA><<<grid, ch_threads(64), chain_smem<SIGMA>(t), st>>>(a); break;
  }
}

size_t pairs_smem(int max_n) {
  const size_t n = max_n, np = n * (n + 1) / 2;
  return (2 * n * n + np * (np | 1)) * sizeof(double2);
}
size_t sigma_smem(int max_np) { return std::max((size_t)max_np * max_np, (size_t)256) * sizeof(double2); }

bool up(void** dst, const void* src, size_t bytes) {
  if (cudaMalloc(dst, bytes ? bytes : 16) != cudaSuccess) {
    *dst = nullptr;
    cudaGetLastError();
    return false;
  }
  return !src || cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice) == cudaSuccess;
}

gw_status launch_status(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) return GW_OK;
  set_last_error(std::string(what) + ": " + cudaGetErrorString(e));
  return GW_ERR_CUDA;
}

}  // namespace

// The chain takes C symmetric in (L, L'') with at most 64 product functions and 64 pairs
// (n <= 10) per species while a unit's digits and both static operands fit shared memory
// (n = 9 up to K = 64, n = 10 up to K = 32); any other plan keeps k_polarizability_fp64 /
// k_self_energy_fp64 with one digit product, and so do small bases: a unit costs the chain
// the same for any K <= 16 and n <= 5, and the other path less and less.  8-atom cell, 2x2x2 k,
// 48 nodes, chain against the other path, P and Sigma in us: n = 4 K = 16 258 / 160 and 537 /
// 398, K = 32 333 / 372 and 681 / 894; n = 5 K = 16 267 / 267 and 559 / 598; n = 9 K = 8 529 /
// 521 and 1257 / 1046, K = 16 541 / 977 and 1284 / 2057, K = 64 907 / 4122 and 1880 / 9605.
constexpr int kChainMinK = 12, kChainMinKnn = 400;
void chain_init(ChainPlan& c, const HostPlan& h) {
  c = ChainPlan{};
  if (!h.c_symmetric) return;
  int max_k = 0, max_np = 0, max_n = 0;
  for (int s = 0; s < h.n_species; ++s) {
    max_n = std::max(max_n, h.n_orb[s]);
    max_k = std::max(max_k, h.n_prod[s]);
  }
  max_np = max_n * (max_n + 1) / 2;
  if (max_k > kChainMax || max_np > kChainMax) return;
  if (max_k < kChainMinK || max_k * max_n * max_n < kChainMinKnn) return;
  c.max_pairs = max_np;
  c.kp.NT = (max_k + 15) / 16 * 16;
  c.kp.KS = (max_np + 15) / 16;
  c.pk.NT = (max_np + 15) / 16 * 16;
  c.pk.KS = (max_k + 15) / 16;
  int dev = 0, smem_max = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&c.n_sm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const size_t lim = (size_t)std::max(smem_max, 0) - 2048;  // the kernel's static shared memory
  if (chain_smem<false>(c.kp) > lim || chain_smem<true>(c.pk) > lim || pairs_smem(max_n) > lim) return;
  std::vector<unsigned char> pr((size_t)h.n_species * 2 * kChainMax, 0), pi((size_t)h.n_species * 256, 0);
  for (int s = 0; s < h.n_species; ++s) {
    const int n = h.n_orb[s];
    int p = 0;
    auto add = [&](int i, int j) {
      pr[(size_t)s * 2 * kChainMax + p] = (unsigned char)i;
      pr[(size_t)s * 2 * kChainMax + kChainMax + p] = (unsigned char)j;
      pi[(size_t)s * 256 + i * 16 + j] = pi[(size_t)s * 256 + j * 16 + i] = (unsigned char)p;
      ++p;
    };
    for (int i = 0; i < n; ++i) add(i, i);
    for (int i = 0; i < n; ++i)
      for (int j = i + 1; j < n; ++j) add(i, j);
  }
  auto table = [&](ChainTable& t, bool rows_k) -> bool {
    const size_t per = (size_t)t.KS * kOzDigits * t.NT * 16;  // uint16 per species
    std::vector<uint16_t> dig(per * h.n_species, 0);
    std::vector<int> ex((size_t)t.NT * h.n_species, 0);
    for (int s = 0; s < h.n_species; ++s) {
      const int n = h.n_orb[s], np = n * (n + 1) / 2, K = h.n_prod[s];
      const int rows = rows_k ? K : np, red = rows_k ? np : K;
      auto value = [&](int r, int k) {
        const int kk = rows_k ? r : k, p = rows_k ? k : r;
        const unsigned char* q = &pr[(size_t)s * 2 * kChainMax];
        return h.C[s][((size_t)kk * n + q[p]) * n + q[kChainMax + p]];
      };
      for (int r = 0; r < rows; ++r) {
        int mx = 0;
        for (int k = 0; k < red; ++k) mx = std::max(mx, host_exp_field(value(r, k)));
        const int e = mx > 0 ? mx - 1022 : 0;
        ex[(size_t)s * t.NT + r] = e;
        t.e_min = std::min(t.e_min, e);
        t.e_max = std::max(t.e_max, e);
        for (int k = 0; k < red; ++k) {
          uint16_t d[kOzDigits];
          host_tf_digits(host_fixed56(value(r, k), e), d);
          const size_t at = s * per + (size_t)(k / 16) * kOzDigits * t.NT * 16 + umma::kmajor_offset(t.NT, r, k % 16) / 2;
          for (int q = 0; q < kOzDigits; ++q) dig[at + (size_t)q * t.NT * 16] = d[q];
        }
      }
    }
    return up((void**)&t.d_B, dig.data(), dig.size() * sizeof(uint16_t)) &&
           up((void**)&t.d_e, ex.data(), ex.size() * sizeof(int));
  };
  if (!table(c.kp, true) || !table(c.pk, false) || !up((void**)&c.d_pair, pr.data(), pr.size()) ||
      !up((void**)&c.d_pidx, pi.data(), pi.size()) ||
      !up((void**)&c.d_species, h.species.data(), h.species.size() * sizeof(int))) {
    chain_free(c);
    return;
  }
  if (chain_raise<false>(c.kp) != cudaSuccess || chain_raise<true>(c.pk) != cudaSuccess ||
      raise_smem_limit(k_polarizability_pairs, pairs_smem(max_n)) != cudaSuccess ||
      raise_smem_limit(k_sigma_pairs, sigma_smem(max_np)) != cudaSuccess) {
    cudaGetLastError();
    chain_free(c);
    return;
  }
  c.ok = true;
}

void chain_free(ChainPlan& c) {
  void* ptrs[] = {c.kp.d_B, c.kp.d_e, c.pk.d_B, c.pk.d_e, c.d_pair, c.d_pidx, c.d_species,
                  c.d_AP, c.d_eP, c.d_AS, c.d_eS, c.d_D};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  c = ChainPlan{};
}

gw_status chain_alloc_p(ChainPlan& c, const HostPlan& h, size_t cap) {
  const size_t E = (size_t)h.n_entries(), per = c.kp.KS * kChStep + 128 * sizeof(int);
  c.tau_p = (int)std::max<size_t>(1, std::min<size_t>((size_t)(h.n_tau + 1) / 2, cap / std::max<size_t>(1, E * per)));
  const size_t n = E * c.tau_p;
  if (!up((void**)&c.d_AP, nullptr, n * c.kp.KS * kChStep) || !up((void**)&c.d_eP, nullptr, n * 128 * sizeof(int))) {
    cudaFree(c.d_AP);
    c.d_AP = nullptr;
    return GW_ERR_OOM;
  }
  c.p_ready = true;
  return GW_OK;
}

gw_status chain_alloc_s(ChainPlan& c, const HostPlan& h, size_t cap) {
  const size_t E = (size_t)h.n_entries();
  const size_t per = c.pk.KS * kChStep + 128 * sizeof(int) + (size_t)c.max_pairs * 128 * sizeof(double);
  c.tau_s = (int)std::max<size_t>(1, std::min<size_t>((size_t)h.n_tau, cap / std::max<size_t>(1, E * per)));
  const size_t n = E * c.tau_s;
  if (!up((void**)&c.d_AS, nullptr, n * c.pk.KS * kChStep) || !up((void**)&c.d_eS, nullptr, n * 128 * sizeof(int)) ||
      !up((void**)&c.d_D, nullptr, n * c.max_pairs * 128 * sizeof(double))) {
    cudaFree(c.d_AS);
    cudaFree(c.d_eS);
    c.d_AS = nullptr;
    c.d_eS = nullptr;
    return GW_ERR_OOM;
  }
  c.s_ready = true;
  return GW_OK;
}

gw_status chain_polarizability(ChainPlan& c, const HostPlan& h, const DevEntry* d_ent, const double2* G, double2* P,
                               int* d_status, cudaStream_t st) {
  const int nodes = (h.n_tau + 1) / 2;  // C symmetric: the mirrored nodes follow
  int max_n = 0;
  for (int s = 0; s < h.n_species; ++s) max_n = std::max(max_n, h.n_orb[s]);
  for (int s0 = 0; s0 < nodes; s0 += c.tau_p) {
    const int te = std::min(c.tau_p, nodes - s0);
    {
      // the name of the row's FP64 stage on the other path, which is what timings of the row look for
      TimedLaunch tl_("k_polarizability_fp64", st);
      k_polarizability_pairs<<<dim3(h.n_entries(), te), 256, pairs_smem(max_n), st>>>(
          d_ent, c.d_species, c.d_pair, G, h.n_tau, s0, c.kp.KS, c.d_AP, c.d_eP);
    }
    ChainArgs a{};
    a.ent = d_ent;
    a.species = c.d_species;
    a.n_units = h.n_entries() * te;
    a.tau_eff = te;
    a.KS = c.kp.KS;
    a.Adig = c.d_AP;
    a.eA = c.d_eP;
    a.B = c.kp.d_B;
    a.eB = c.kp.d_e;
    a.eB_min = c.kp.e_min;
    a.eB_max = c.kp.e_max;
    a.P = P;
    a.n_tau = h.n_tau;
    a.s0 = s0;
    a.ms_shift = h.spin == 2 ? 1 : 0;
    a.status = d_status;
    chain_launch<false>(c.kp, a, c.n_sm, st);
    const gw_status e = launch_status("FP64 polarizability");
    if (e != GW_OK) return e;
  }
  return GW_OK;
}

gw_status chain_self_energy(ChainPlan& c, const HostPlan& h, const DevEntry* d_ent, const double2* G, const double2* W,
                            int n_slices, int g_fixed, double sign, double2* Sig, int* d_status, cudaStream_t st) {
  for (int s0 = 0; s0 < n_slices; s0 += c.tau_s) {
    const int te = std::min(c.tau_s, n_slices - s0);
    {
      TimedLaunch tl_("k_slice_w_units", st);
      k_slice_w_units<<<dim3(h.n_entries(), te), 256, 0, st>>>(d_ent, W, n_slices, s0, c.pk.KS, c.d_AS, c.d_eS);
    }
    ChainArgs a{};
    a.ent = d_ent;
    a.species = c.d_species;
    a.n_units = h.n_entries() * te;
    a.tau_eff = te;
    a.KS = c.pk.KS;
    a.Adig = c.d_AS;
    a.eA = c.d_eS;
    a.B = c.pk.d_B;
    a.eB = c.pk.d_e;
    a.eB_min = c.pk.e_min;
    a.eB_max = c.pk.e_max;
    a.D = c.d_D;
    a.ld_d = c.max_pairs;
    a.status = d_status;
    chain_launch<true>(c.pk, a, c.n_sm, st);
    {
      TimedLaunch tl_("k_sigma_pairs", st);
      k_sigma_pairs<<<dim3(h.n_entries(), te), 256, sigma_smem(c.max_pairs), st>>>(
          d_ent, c.d_species, c.d_pidx, c.d_D, c.max_pairs, G, h.n_tau, g_fixed, s0, sign, Sig, n_slices);
    }
    const gw_status e = launch_status("FP64 self-energy");
    if (e != GW_OK) return e;
  }
  return GW_OK;
}

}  // namespace gw
