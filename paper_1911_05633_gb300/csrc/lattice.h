// Lattice transforms R <-> k by FP64-accurate digit products, for meshes with general phases
// (kernels_lattice.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace gw {

constexpr int kLatMaxK = 32;                          // mesh points (reductions of at most 64 terms)
constexpr int kLatHeld = 8;                           // mesh points whose values or sums the FP64 kernels hold in registers
constexpr size_t kLatMaxBytes = (size_t)64 << 20;     // operands of all pairs, per direction

struct LatticePlan {
  bool ok = false;
  int n_active = 0, max_cls = 0, n_sm = 0;
  bool all_pairs = false;          // every ordered pair has an entry
  double sweep[2] = {0.0, 0.0};    // per kind (orbital, product) and element of the pairs: elements that the FP64 kernels' warps visit
  int* d_first = nullptr;          // [n_active + 1] entry ranges
  // [0]: k -> R, [1]: R -> k
  uint16_t* d_B[2] = {nullptr, nullptr};
  long long* d_off[2] = {nullptr, nullptr};
  int* d_e[2] = {nullptr, nullptr};
};

// ok where the plan's transforms fit and their operands are on the device.
void lattice_init(LatticePlan& l, const HostPlan& h);
// Whether a transform of n_slices slices goes to the tensor cores.
bool lattice_takes(const LatticePlan& l, const HostPlan& h, bool pb, int n_slices, bool to_k);
void lattice_free(LatticePlan& l);
// dense [n_k][n_slices][N][N] <-> the entry layout with n_slices slices.
gw_status lattice_run(const LatticePlan& l, const HostPlan& h, const DevEntry* d_ent, const int* d_row_off,
                      const double2* d_phase, bool pb, int n_slices, bool to_k, double2* dense, double2* entries,
                      int* d_status, cudaStream_t st);

}  // namespace gw
