// Batches of small dense complex FP64 matrices (kernels_gj.cu): Gauss-Jordan inverses in
// shared memory, and traces of shifted inverses through the Hessenberg form.
#pragma once

#include <cuda_runtime.h>

namespace gw {

// The largest order held in shared memory: N (N | 1) complex values and the vectors.
constexpr int kGJSmemMax = 112;
// The largest order of the trace kernel: a block holds four rows of each of 4 matrices.
constexpr int kHessMaxN = 880;

// Dynamic shared-memory opt-in of the inverse for order N (call with the device current).
cudaError_t gj_setup(int N, bool columns = false);
// In-place inverses of `batch` N x N matrices; perm: [batch][N] scratch (read only above
// kGJSmemMax, where `columns` asks for the form without panels).  A zero pivot sets *status.
void gj_batch(double2* mats, int* perm, int batch, int N, long long stride, int* status, cudaStream_t st,
              bool columns = false);

// The panel form on the matrices with only[b] != 0 (N up to 430; the others are not touched).
cudaError_t gj_only_setup(int N);
void gj_batch_only(double2* mats, int* perm, int batch, int N, int* status, const int* only, cudaStream_t st);

cudaError_t hess_setup(int N);
// out[b] = Hessenberg form of i w_n - H(k) - Sx(k) - Sc(k, n), b = k n_w + n (Sx, Sc may be
// null); scale[b]: the largest |re| + |im| of the matrix.
void hess_reduce(const double2* H, const double2* Sx, const double2* Sc, const double* w, int N, int n_w,
                 long long n_b, double2* out, double* scale, cudaStream_t st);
// tr[b] = tr (mu + Hs[b])^{-1}; *flag set where a pivot is too small for that.
void hess_trace(const double2* Hs, const double* scale, double mu, int N, long long n_b, double2* tr, int* flag,
                cudaStream_t st);

}  // namespace gw
