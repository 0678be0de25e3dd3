// FP64 P and Sigma contractions (Eqs. P_MM and S_MM) over symmetric orbital pairs, as two
// chained FP64-accurate digit products per unit on the tensor cores (kernels_chain.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace gw {

constexpr int kChainMax = 64;  // product functions per atom and orbital pairs n (n + 1) / 2 at most

// A static column operand per species: digits [KS][kOzDigits][NT x 16] and exponents [NT].
struct ChainTable {
  int KS = 0, NT = 0;
  int e_min = 0, e_max = 0;  // of the exponents
  uint16_t* d_B = nullptr;  // [n_species] operands, back to back
  int* d_e = nullptr;       // [n_species][NT]
};

struct ChainPlan {
  bool ok = false;            // the plan's species fit (and C is symmetric)
  ChainTable kp;              // rows K, reduction over pairs: C[K][pair]   (both products of P)
  ChainTable pk;              // rows pair, reduction over K: C[K][pair]    (both products of Sigma)
  unsigned char* d_pair = nullptr;  // [n_species][2][kChainMax]: L and L'' of each pair
  unsigned char* d_pidx = nullptr;  // [n_species][16 x 16]: pair of (L, L'')
  int* d_species = nullptr;   // [n_atoms]
  int n_sm = 0;
  int max_pairs = 0;
  // per contraction: the digits of one pass's units, their row exponents, slices per pass
  bool p_ready = false, s_ready = false;
  uint16_t* d_AP = nullptr;
  int* d_eP = nullptr;
  int tau_p = 0;
  uint16_t* d_AS = nullptr;
  int* d_eS = nullptr;
  double* d_D = nullptr;      // Sigma: [units][max_pairs][128] second product of one pass
  int tau_s = 0;
};

// Whether the plan's contractions fit; uploads the tables when they do (ok: false as well when
// there is no memory for them).
void chain_init(ChainPlan& c, const HostPlan& h);
// Scratch of one contraction within `cap` bytes (p_ready, s_ready).
gw_status chain_alloc_p(ChainPlan& c, const HostPlan& h, size_t cap);
gw_status chain_alloc_s(ChainPlan& c, const HostPlan& h, size_t cap);
void chain_free(ChainPlan& c);
// P of every entry and computed node (and the mirrored nodes).
gw_status chain_polarizability(ChainPlan& c, const HostPlan& h, const DevEntry* d_ent, const double2* G, double2* P,
                               int* d_status, cudaStream_t st);
// sign * Sigma for n_slices slices of W (g_fixed >= 0: that slice of G for every one).
gw_status chain_self_energy(ChainPlan& c, const HostPlan& h, const DevEntry* d_ent, const double2* G, const double2* W,
                            int n_slices, int g_fixed, double sign, double2* Sig, int* d_status, cudaStream_t st);

}  // namespace gw
