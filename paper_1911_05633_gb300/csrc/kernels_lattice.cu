// Lattice transforms R <-> k (Sec. 2) on meshes whose phases are not all quarter turns, as
// FP64-accurate digit products on the tensor cores.  For one ordered atom pair (a, b) the
// transform is a small matrix over the pair's classes and the mesh,
//   k -> R:  F_R[class]  = (1/N_k) sum_k conj(e^{ik.R}) F_k,   reduction (k, Re/Im)
//   R -> k:  F_k         = sum_class e^{ik.R} F_R[class],      reduction (class, Re/Im)
// applied to every (slice, i, j) of the pair's block: rows of a GEMM whose small operand
// (<= 64 x 64, digits made once per plan) is one per pair.
//
// In FP64 arithmetic a term is four multiply-adds and the chip issues two per clock and SM:
// 27 points and 5.4 kept classes per pair take 290 clocks per element and SM.  Cutting the 54
// values into digits and reading the sums back is integer and FP32 work of about a tenth of
// that, and the products are free beside it.
// G, v and Sigma of the 16-atom cell on a 3x3x3 mesh (1392 entries, 48 slices): 0.98 ms in
// three launches, 4.64 ms by k_gather_k_to_R and k_scatter_R_to_k.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <vector>

#include "kernels.h"
#include "ktimer.h"
#include "lattice.h"
#include "ozdigits.h"
#include "smem_limit.h"

namespace gw {

namespace {

constexpr uint64_t kLtWaitNs = 500ull * 1000ull * 1000ull;
constexpr int kLtWarps = 8;                           // slicer warps, and as many epilogue warps
constexpr int kLtThreads = 32 * (2 * kLtWarps + 1);   // and one that issues the products
constexpr int kLtStages = 3;
constexpr uint32_t kLtStep = kOzDigits * kTfPlane;    // 32 KB: digits of 128 rows, one K step
// Rows that the digits hold: the largest exponent field of a row within these.  A sum is a
// multiple of 2^(e - 61) for the row's scale 2^e (2^-56 of it times the smallest column scale,
// 2^-5 at 32 points) and below 2^(e + 7), so that these keep it a normal double, and what the
// digits drop of such a row, its subnormal values, is below 2^-62 of it.  Any other row that
// is not all zero (G(tau) far from both ends at low temperature; a NaN or an infinity, which
// the digits would lose) is summed in FP64 once its block's tiles are done: taken within the
// read-out, or told from zero rows by the slicers, such rows cost transforms without any 1.4 %
// in the middle and up to 6 % (launches of 20 to 45 us).
constexpr int kLtLow = 64, kLtHigh = 2032;
constexpr int kLtDirect = 1 << 20;                    // in place of such a row's scale exponent

struct LatArgs {
  const DevEntry* ent;
  const int* pair_first;   // [n_active + 1] entry range of each pair with entries
  const int* row_off;      // atoms' offsets in the dense matrix
  int pb, n_k, n_slices, ld;
  long long k_stride, s_stride;  // of the dense side
  double2* dense;
  double2* entries;
  const uint16_t* B;       // static operands
  const long long* B_off;  // [n_active] offset of a pair's operand (uint16 units)
  const int* eB;           // [n_active][64]
  const double2* phase;    // [E][n_k] e^{+i k.R}
  double scale;            // 1 / N_k
  int tiles_per_block;
  int* status;
};

// Columns of a pair's operand, padded to the MMA's multiple of 16.
__host__ __device__ inline int lat_nt(int cols) { return (cols + 15) & ~15; }

// A pair's classes in shared memory, its first entry and the sizes of its transform.
struct LatPair {
  const long long* off;
  const int* re;
  const int* ce;
  int e0, n_in, n_out;
};

// Outputs m0 .. m0 + 7 of one row as k_gather_k_to_R and k_scatter_R_to_k take them.  G of 16
// atoms on 3x3x3, 48 slices, of which 0 / 8 / 24 / 48 are below 1e-290 everywhere: k -> R 0.45 /
// 0.78 / 1.33 / 2.34 ms, 1.80 by k_gather_k_to_R; R -> k 0.27 / 0.50 / 0.95 / 1.70, 1.96.
template <bool SCATTER>
__device__ __forceinline__ void lat_direct(const LatArgs& g, const LatPair p, long long el, int s, int i, int j, int m0) {
#pragma unroll 1
  for (int m = m0; m < min(m0 + 8, p.n_out); ++m) {
    if (!SCATTER && !(i < p.re[m] && j < p.ce[m])) continue;
    double2 a = make_double2(0.0, 0.0);
#pragma unroll 4
    for (int q = 0; q < p.n_in; ++q) {
      if (SCATTER && !(i < p.re[q] && j < p.ce[q])) continue;
      const double2 v = SCATTER ? g.entries[p.off[q] + (long long)s * p.re[q] * p.ce[q] + i * p.ce[q] + j]
                                : g.dense[q * g.k_stride + el];
      const double2 f = g.phase[(long long)(p.e0 + (SCATTER ? q : m)) * g.n_k + (SCATTER ? m : q)];
      const double fy = SCATTER ? f.y : -f.y;
      a = make_double2(fma(f.x, v.x, fma(-fy, v.y, a.x)), fma(f.x, v.y, fma(fy, v.x, a.y)));
    }
    if (SCATTER) g.dense[m * g.k_stride + el] = a;
    else g.entries[p.off[m] + (long long)s * p.re[m] * p.ce[m] + i * p.ce[m] + j] =
             make_double2(a.x * g.scale, a.y * g.scale);
  }
}

// Block (pair, chunk of its row tiles).  Slicer warps hold their row's values (all loads in
// flight at once), take the row's scale and cut them; the epilogue reads the level sums as
// exact integers.  Two sets of accumulators where they fit (up to 32 columns).
template <int KS, bool SCATTER>
__global__ void __launch_bounds__(kLtThreads, 1) k_lattice_tc(const __grid_constant__ LatArgs g) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint32_t tmem_base;
  __shared__ __align__(8) uint64_t a_full[kLtStages], a_empty[kLtStages];
  __shared__ __align__(8) uint64_t t_full[2], t_empty[2], b_full, drained;
  __shared__ __align__(8) uint64_t e_full[2], e_empty[2];
  __shared__ int eA_s[2][128];
  __shared__ int eB_s[64];
  __shared__ long long off_s[32];  // first element of each class's entry
  __shared__ int re_s[32], ce_s[32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int e0 = g.pair_first[blockIdx.x], n_cls = g.pair_first[blockIdx.x + 1] - e0;
  const DevEntry E0 = g.ent[e0];
  const int ro = g.row_off[E0.a], co = g.row_off[E0.b];
  const int ra = g.row_off[E0.a + 1] - ro, cb = g.row_off[E0.b + 1] - co, blk = ra * cb;  // the full block
  const long long rows = (long long)blk * g.n_slices;
  const int n_tiles = (int)((rows + 127) / 128);
  const int t0 = blockIdx.y * g.tiles_per_block, t1 = min(n_tiles, t0 + g.tiles_per_block);
  if (t0 >= t1) return;
  const int n_in = SCATTER ? n_cls : g.n_k, n_out = SCATTER ? g.n_k : n_cls;
  const int NT = lat_nt(2 * n_out);
  const int n_ks = (2 * n_in + 15) / 16;  // <= KS
  const int n_buf = NT <= 32 ? 2 : 1;
  const uint32_t BK = (uint32_t)kOzDigits * NT * 32;
  unsigned char* Bs = sm;
  unsigned char* As = sm + n_ks * BK;
  if (warp == kLtWarps) {
    tmem_alloc(&tmem_base, 512);
    tmem_relinquish();
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < kLtStages; ++s) {
      mbar_init(&a_full[s], 32 * kLtWarps);
      mbar_init(&a_empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&e_full[b], 32 * kLtWarps);
      mbar_init(&e_empty[b], 32 * kLtWarps);
      mbar_init(&t_full[b], 1);
      mbar_init(&t_empty[b], 32 * kLtWarps);
    }
    mbar_init(&b_full, 1);
    mbar_init(&drained, 1);
    fence_mbar_init();
  }
  if (threadIdx.x < 64) eB_s[threadIdx.x] = g.eB[blockIdx.x * 64 + threadIdx.x];
  if (threadIdx.x < n_cls) {
    const DevEntry& E = g.ent[e0 + threadIdx.x];
    off_s[threadIdx.x] = (g.pb ? E.off_pb : E.off_orb) * g.n_slices;
    re_s[threadIdx.x] = g.pb ? E.Ka : E.na;
    ce_s[threadIdx.x] = g.pb ? E.Kb : E.nb;
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tm = tmem_base;
  // element (slice, i, j) of row x: place in the dense matrix, and in an entry's block
  auto dense_at = [&](int s, int i, int j) {
    return (long long)s * g.s_stride + (long long)(ro + i) * g.ld + co + j;
  };
  // value m (mesh point or class) of a row
  auto value = [&](int m, int s, int i, int j) {
    if (!SCATTER) return __ldg(g.dense + m * g.k_stride + dense_at(s, i, j));
    if (i < re_s[m] && j < ce_s[m])
      return __ldg(g.entries + off_s[m] + (long long)s * re_s[m] * ce_s[m] + i * ce_s[m] + j);
    return make_double2(0.0, 0.0);
  };
  bool ok = true;
  if (warp < kLtWarps) {
    const int r = 16 * warp + (lane & 15), h = lane >> 4;
    int step = 0;
    for (int t = t0; t < t1 && ok; ++t) {
      const long long x = (long long)t * 128 + r;
      const bool valid = x < rows;
      const int s = valid ? (int)(x / blk) : 0, ij = valid ? (int)(x - (long long)s * blk) : 0;
      const int i = ij / cb, j = ij - i * cb;
      double w[KS][8];
      int mx = 0;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int m = ks * 8 + 4 * h + q;  // mesh point or class
          double2 v = make_double2(0.0, 0.0);
          if (valid && m < n_in) v = value(m, s, i, j);
          w[ks][2 * q] = v.x;
          w[ks][2 * q + 1] = v.y;
        }
#pragma unroll
      for (int ks = 0; ks < KS; ++ks)
#pragma unroll
        for (int u = 0; u < 8; ++u) mx = max(mx, exp_field(w[ks][u]));
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
      const int e = mx > 0 ? mx - 1022 : 0;
      const int it = t - t0, b = it & 1;
      ok = mbar_wait(&e_empty[b], (uint32_t)((it >> 1) & 1) ^ 1u, kLtWaitNs, g.status);
      if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
      if (h == 0) eA_s[b][r] = mx < kLtLow || mx > kLtHigh ? kLtDirect : e;
      mbar_arrive(&e_full[b]);
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        if (ks < n_ks && ok) {
          const int st = step % kLtStages;
          ok = mbar_wait(&a_empty[st], (uint32_t)((step / kLtStages) & 1) ^ 1u, kLtWaitNs, g.status);
          ok = __all_sync(0xffffffffu, ok);
          if (ok) {
            unsigned char* A = As + st * kLtStep + kmajor_offset(128, r, 8 * h);
            long long M[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) M[u] = fixed56(w[ks][u], e);
            tf_cut8(M, A);
            fence_smem_to_async();
            mbar_arrive(&a_full[st]);
            ++step;
          }
        }
      }
    }
    if (!ok) atomicExch(g.status, 2);
  } else if (warp == kLtWarps) {
    if (lane == 0) {
      const uint32_t a_base = smem_u32(As), b_base = smem_u32(Bs);
      const unsigned char* src = reinterpret_cast<const unsigned char*>(g.B + g.B_off[blockIdx.x]);
      mbar_arrive_expect_tx(&b_full, n_ks * BK);
      for (int ks = 0; ks < n_ks; ++ks) bulk_g2s(Bs + ks * BK, src + (size_t)ks * BK, BK, &b_full);
      ok = mbar_wait(&b_full, 0, kLtWaitNs, g.status);
      int step = 0;
      for (int t = t0; t < t1 && ok; ++t) {
        const int it = t - t0, bf = n_buf == 2 ? it & 1 : 0, use = n_buf == 2 ? it >> 1 : it;
        if (!(ok = mbar_wait(&t_empty[bf], (uint32_t)(use & 1) ^ 1u, kLtWaitNs, g.status))) break;
        fence_after_sync();
        for (int ks = 0; ks < n_ks; ++ks, ++step) {
          const int st = step % kLtStages;
          if (!(ok = mbar_wait(&a_full[st], (uint32_t)((step / kLtStages) & 1), kLtWaitNs, g.status))) break;
          fence_after_sync();
          tf_issue(NT, tm + (uint32_t)(bf * 256), smem_desc(a_base + st * kLtStep, 128, 256),
                   smem_desc(b_base + ks * BK, 128, 256), ks == 0);
          mma_commit(&a_empty[st]);
        }
        if (ok) mma_commit(&t_full[bf]);
      }
      // every product issued has finished before the accumulators are released
      mma_commit(&drained);
      if (!mbar_wait(&drained, 0, kLtWaitNs, nullptr)) ok = false;
      if (!ok) {
        atomicExch(g.status, 2);
        mbar_wait(&b_full, 0, kLtWaitNs, nullptr);
      }
    }
  } else {
    const int q = warp & 3, half = (warp - kLtWarps - 1) >> 2;
    const int row = 32 * q + lane, n_chunks = NT / 16;
    unsigned long long left = 0;  // tiles (modulo 64) where this thread's row was not for the digits
    // rows beyond every class's block are zero
    const int r_max = SCATTER ? __reduce_max_sync(0xffffffffu, lane < n_cls ? re_s[lane] : 0) : ra;
    const int c_max = SCATTER ? __reduce_max_sync(0xffffffffu, lane < n_cls ? ce_s[lane] : 0) : cb;
    for (int t = t0; t < t1 && ok; ++t) {
      const int it = t - t0, b = it & 1, bf = n_buf == 2 ? it & 1 : 0, use = n_buf == 2 ? it >> 1 : it;
      const long long x = (long long)t * 128 + row;
      const bool valid = x < rows;
      const int s = valid ? (int)(x / blk) : 0, ij = valid ? (int)(x - (long long)s * blk) : 0;
      const int i = ij / cb, j = ij - i * cb;
      ok = mbar_wait(&e_full[b], (uint32_t)((it >> 1) & 1), kLtWaitNs, g.status);
      if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
      const int ea = eA_s[b][row];
      if (ea == kLtDirect && valid && i < r_max && j < c_max && half < n_chunks) left |= 1ull << (it & 63);
      mbar_arrive(&e_empty[b]);
      ok = mbar_wait(&t_full[bf], (uint32_t)(use & 1), kLtWaitNs, g.status);
      if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
      fence_after_sync();
      const uint32_t taddr = tm + (uint32_t)(bf * 256) + ((uint32_t)(32 * q) << 16);
      int last = half;  // this warp's last chunk (none: released at once)
      while (last + 2 < n_chunks) last += 2;
      if (half >= n_chunks) {
        fence_before_sync();
        mbar_arrive(&t_empty[bf]);
      }
      for (int c = half; c < n_chunks; c += 2) {
        long long S[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) S[k] = 0;
#pragma unroll
        for (int l = 0; l < 8; l += 2) {
          float v[32];
          tmem_ld16x2(taddr + (uint32_t)(l * NT + 16 * c), (uint32_t)NT, v);
          const float s0 = __int_as_float((127 + 7 * l) << 23), s1 = __int_as_float((127 + 7 * (l + 1)) << 23);
#pragma unroll
          for (int k = 0; k < 16; ++k) {  // units of 2^-56 of the scale (64 terms: below 64 of it)
            const int P = tf_pair_int<false>(v[k], s0, v[16 + k], s1);
            if (l < 6) S[k] += (long long)P << (42 - 7 * (l + 1));
            else S[k] += (long long)((P + 64) >> 7);
          }
        }
        if (c == last) {
          fence_before_sync();
          mbar_arrive(&t_empty[bf]);
        }
        if (!valid) continue;
#pragma unroll
        for (int k = 0; k < 16; k += 2) {
          const int n = 16 * c + k, m = n >> 1;
          if (m >= n_out) break;
          const double2 z = make_double2(tf_i2d(S[k], ea + eB_s[n] - 56), tf_i2d(S[k + 1], ea + eB_s[n + 1] - 56));
          if (SCATTER) g.dense[m * g.k_stride + dense_at(s, i, j)] = z;
          else if (i < re_s[m] && j < ce_s[m])
            g.entries[off_s[m] + (long long)s * re_s[m] * ce_s[m] + i * ce_s[m] + j] = z;
        }
      }
    }
    if (!ok) atomicExch(g.status, 2);
    // what the digits could not hold, over what was written for it (zeros: right already)
    for (int t = t0; left && ok && t < t1; ++t) {
      const long long x = (long long)t * 128 + row;
      if (x >= rows) break;
      if (!((left >> ((t - t0) & 63)) & 1ull)) continue;
      const int s = (int)(x / blk), ij = (int)(x - (long long)s * blk), i = ij / cb, j = ij - i * cb;
      unsigned long long any = 0;
      int mx = 0;
#pragma unroll 4
      for (int m = 0; m < n_in; ++m) {
        const double2 v = value(m, s, i, j);
        mx = max(mx, max(exp_field(v.x), exp_field(v.y)));
        any |= (unsigned long long)(__double_as_longlong(v.x) | __double_as_longlong(v.y)) << 1;
      }
      if (any == 0 || (mx >= kLtLow && mx <= kLtHigh)) continue;
      for (int c = half; c < n_chunks; c += 2)
        lat_direct<SCATTER>(g, LatPair{off_s, re_s, ce_s, e0, n_in, n_out}, dense_at(s, i, j), s, i, j, 8 * c);
    }
  }
  fence_before_sync();
  __syncthreads();
  if (warp == kLtWarps) tmem_dealloc(tm, 512);
}

size_t lat_smem(int KS, int NT) {
  // more than half of the SM's shared memory: one block per SM (all 512 tensor-memory columns)
  return std::max((size_t)KS * kOzDigits * NT * 32 + (size_t)kLtStages * kLtStep, (size_t)116 * 1024);
}

template <bool SCATTER>
cudaError_t lat_raise() {
  cudaError_t e = raise_smem_limit(k_lattice_tc<1, SCATTER>, lat_smem(1, 64));
  if (e == cudaSuccess) e = raise_smem_limit(k_lattice_tc<2, SCATTER>, lat_smem(2, 64));
  if (e == cudaSuccess) e = raise_smem_limit(k_lattice_tc<3, SCATTER>, lat_smem(3, 64));
  if (e == cudaSuccess) e = raise_smem_limit(k_lattice_tc<4, SCATTER>, lat_smem(4, 64));
  return e;
}
template <bool SCATTER>
void lat_launch(int KS, dim3 grid, size_t smem, const LatArgs& a, cudaStream_t st) {
  TimedLaunch tl_("k_lattice_tc", st);
  switch (KS) {
    case 1: k_lattice_tc<1, SCATTER><<<grid, kLtThreads, smem, st>>>(a); break;
    case 2: k_lattice_tc<2, SCATTER><<<grid, kLtThreads, smem, st>>>(a); break;
    case 3: k_lattice_tc<3, SCATTER><<<grid, kLtThreads, smem, st>>>(a); break;
    default: k_lattice_tc<4, SCATTER><<<grid, kLtThreads, smem, st>>>(a); break;
  }
}

// Elements (lane, class) that the warps of k_gather_k_to_R and k_scatter_R_to_k go through for
// one slice, per element of the pairs with entries: a warp takes 32 consecutive elements of a
// row atom's band, and all its lanes wait for the one with the most classes.
double lat_sweep(const HostPlan& h, const std::vector<int>& ro) {
  const int n = h.n_atoms, N = ro[n];
  std::vector<int> cls(N);  // of the pair that each column belongs to
  double steps = 0.0, el = 0.0;
  for (int a = 0; a < n; ++a) {
    for (int b = 0; b < n; ++b)
      for (int i = ro[b]; i < ro[b + 1]; ++i) cls[i] = h.pair_start[a * n + b + 1] - h.pair_start[a * n + b];
    const long long band = (long long)(ro[a + 1] - ro[a]) * N;
    int col = 0;
    for (long long x = 0; x < band; x += 32) {
      int most = 0;
      for (long long y = x; y < std::min(band, x + 32); ++y) {
        most = std::max(most, cls[col]);
        el += cls[col] > 0;
        if (++col == N) col = 0;
      }
      steps += 32.0 * most;
    }
  }
  return el > 0.0 ? steps / el : 0.0;
}

}  // namespace

// Taken on meshes of at most 32 points with some phase that is no quarter turn (quarter turns
// cost two additions per term and stay with the FP64 kernels), while the pairs' operands are
// small beside the data.
void lattice_init(LatticePlan& l, const HostPlan& h) {
  l = LatticePlan{};
  std::vector<int> first;
  for (size_t q = 0; q + 1 < h.pair_start.size(); ++q)
    if (h.pair_start[q + 1] > h.pair_start[q]) first.push_back(h.pair_start[q]);
  const int n_act = (int)first.size();
  first.push_back(h.n_entries());
  if (!h.phase_code.empty() || h.n_k > kLatMaxK || n_act == 0) return;
  for (int p = 0; p < n_act; ++p) l.max_cls = std::max(l.max_cls, first[p + 1] - first[p]);
  l.n_active = n_act;
  l.all_pairs = n_act == h.n_atoms * h.n_atoms;
  if (h.n_k <= kLatHeld) {
    l.sweep[0] = lat_sweep(h, h.orb_off);
    l.sweep[1] = lat_sweep(h, h.pb_off);
  }
  for (int d = 0; d < 2; ++d) {  // 0: k -> R, 1: R -> k
    std::vector<long long> off(n_act);
    std::vector<int> ex((size_t)n_act * 64, 0);
    size_t tot = 0;
    for (int p = 0; p < n_act; ++p) {
      const int nc = first[p + 1] - first[p], n_in = d ? nc : h.n_k, n_out = d ? h.n_k : nc;
      off[p] = (long long)tot;
      tot += (size_t)((2 * n_in + 15) / 16) * kOzDigits * lat_nt(2 * n_out) * 16;
    }
    if (tot * sizeof(uint16_t) > kLatMaxBytes) {
      lattice_free(l);
      return;
    }
    std::vector<uint16_t> dig(tot, 0);
    for (int p = 0; p < n_act; ++p) {
      const int nc = first[p + 1] - first[p], n_in = d ? nc : h.n_k, n_out = d ? h.n_k : nc, NT = lat_nt(2 * n_out);
      // out (m, c) from in (q, c'): e^{+-ik.R} as a real 2 x 2 block
      auto value = [&](int n, int k) {
        const int m = n >> 1, q = k >> 1, cls = d ? q : m, kk = d ? m : q;
        const double* ph = &h.phase[2 * ((size_t)(first[p] + cls) * h.n_k + kk)];
        const double f = d ? 1.0 : 1.0 / h.n_k, re = f * ph[0], im = d ? ph[1] : -f * ph[1];
        return (n & 1) == (k & 1) ? re : (n & 1) ? im : -im;
      };
      for (int n = 0; n < 2 * n_out; ++n) {
        int mx = 0;
        for (int k = 0; k < 2 * n_in; ++k) mx = std::max(mx, host_exp_field(value(n, k)));
        const int e = mx > 0 ? mx - 1022 : 0;
        ex[(size_t)p * 64 + n] = e;
        for (int k = 0; k < 2 * n_in; ++k) {
          uint16_t t[kOzDigits];
          host_tf_digits(host_fixed56(value(n, k), e), t);
          const size_t at = off[p] + (size_t)(k / 16) * kOzDigits * NT * 16 + umma::kmajor_offset(NT, n, k % 16) / 2;
          for (int s = 0; s < kOzDigits; ++s) dig[at + (size_t)s * NT * 16] = t[s];
        }
      }
    }
    auto up = [&](void** dst, const void* src, size_t bytes) {
      return cudaMalloc(dst, bytes) == cudaSuccess && cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice) == cudaSuccess;
    };
    if (!up((void**)&l.d_B[d], dig.data(), dig.size() * sizeof(uint16_t)) ||
        !up((void**)&l.d_off[d], off.data(), off.size() * sizeof(long long)) ||
        !up((void**)&l.d_e[d], ex.data(), ex.size() * sizeof(int)) ||
        (d == 0 && !up((void**)&l.d_first, first.data(), first.size() * sizeof(int)))) {
      cudaGetLastError();
      lattice_free(l);  // the FP64 kernels, which need no operands
      return;
    }
  }
  if (lat_raise<false>() != cudaSuccess || lat_raise<true>() != cudaSuccess) {
    cudaGetLastError();
    lattice_free(l);
    return;
  }
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&l.n_sm, cudaDevAttrMultiProcessorCount, dev);
  l.ok = true;
}

// From about 8 million FP64 multiply-adds on, 15 us of the chip; below that either way is launch
// latency.  On up to kLatHeld points the FP64 kernels read an element once for all its classes,
// so that their time is that of the steps their warps take (60 ns per thousand either way),
// while a tile costs this kernel the same for any mesh and class count up to 8 (about 120 ns
// per thousand elements): the line is at 2.2 steps per element k -> R and 1.4 R -> k, where
// the FP64 sum over k of an element is longer.  On 8 atoms, in us FP64 / here: 7x1x1 with 1.25
// classes per pair (1.7 steps) 103 / 184 and 147 / 165, 3x2x1 with 2.6 (2.9) 116 / 103 and
// 113 / 103; 24 atoms with n = 2, 1x3x1, 1.3 classes (3.9) 161 / 82 and 168 / 79.
bool lattice_takes(const LatticePlan& l, const HostPlan& h, bool pb, int n_slices, bool to_k) {
  const double len = (double)(pb ? h.off_pb : h.off_orb).back();
  if (!l.ok || len * n_slices * h.n_k * 4.0 < 8e6) return false;
  return h.n_k > kLatHeld || l.sweep[pb ? 1 : 0] >= (to_k ? 1.4 : 2.2);
}

void lattice_free(LatticePlan& l) {
  for (int d = 0; d < 2; ++d) {
    if (l.d_B[d]) cudaFree(l.d_B[d]);
    if (l.d_off[d]) cudaFree(l.d_off[d]);
    if (l.d_e[d]) cudaFree(l.d_e[d]);
  }
  if (l.d_first) cudaFree(l.d_first);
  l = LatticePlan{};
}

gw_status lattice_run(const LatticePlan& l, const HostPlan& h, const DevEntry* d_ent, const int* d_row_off,
                      const double2* d_phase, bool pb, int n_slices, bool to_k, double2* dense, double2* entries,
                      int* d_status, cudaStream_t st) {
  const std::vector<int>& ro = pb ? h.pb_off : h.orb_off;
  const long long N = ro.back();
  int band = 0;
  for (int a = 0; a < h.n_atoms; ++a) band = std::max(band, ro[a + 1] - ro[a]);
  const long long max_tiles = ((long long)band * band * n_slices + 127) / 128;
  LatArgs a{};
  a.ent = d_ent;
  a.pair_first = l.d_first;
  a.row_off = d_row_off;
  a.pb = pb ? 1 : 0;
  a.n_k = h.n_k;
  a.n_slices = n_slices;
  a.ld = (int)N;
  a.s_stride = N * N;
  a.k_stride = (long long)n_slices * N * N;
  a.dense = dense;
  a.entries = entries;
  a.B = l.d_B[to_k];
  a.B_off = l.d_off[to_k];
  a.eB = l.d_e[to_k];
  a.phase = d_phase;
  a.scale = 1.0 / h.n_k;
  a.status = d_status;
  // about six blocks per SM over the whole launch, at least four tiles each
  const long long want = std::max<long long>(1, 6LL * l.n_sm / l.n_active);
  a.tiles_per_block = (int)std::max<long long>(4, (max_tiles + want - 1) / want);
  const dim3 grid((unsigned)l.n_active, (unsigned)((max_tiles + a.tiles_per_block - 1) / a.tiles_per_block));
  const int n_in = to_k ? l.max_cls : h.n_k, n_out = to_k ? h.n_k : l.max_cls;
  const int KS = (2 * n_in + 15) / 16;
  const size_t smem = lat_smem(KS, lat_nt(2 * n_out));
  if (to_k) {
    // blocks of pairs without entries are zero
    if (!l.all_pairs && cudaMemsetAsync(dense, 0, (size_t)h.n_k * a.k_stride * sizeof(double2), st) != cudaSuccess) {
      set_last_error("R -> k: clearing the dense matrices failed");
      return GW_ERR_CUDA;
    }
    lat_launch<true>(KS, grid, smem, a, st);
  } else {
    lat_launch<false>(KS, grid, smem, a, st);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_last_error(std::string("lattice transform: ") + cudaGetErrorString(e));
    return GW_ERR_CUDA;
  }
  return GW_OK;
}

}  // namespace gw
