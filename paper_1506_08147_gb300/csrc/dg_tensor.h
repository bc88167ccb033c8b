// FP64 contractions of the DG assembly on the tensor cores (dg_tensor.cu).
#pragma once

#include <cuda_runtime.h>

#include <vector>

namespace dgdft {

// out[e][o][r][s] = sum_i A[r][i] in[e][o][i][s], A n_out x n_in row-major
// (element e uses A + e * a_stride), n_out <= 128.  scratch holds
// axis_image_bytes.  *err is set when a bounded device wait ran out.
// shift (NULL, or n_in <= 128 integers per element, A then per element too):
// binary exponents of the inputs' magnitudes; a line's digits count from its
// largest entry, so inputs of different scales enter as in[i] 2^-shift[i], A's
// columns as A[r][i] 2^shift[i].
size_t axis_image_bytes(int n_in, int n_out, int nmat);
cudaError_t launch_axis_tensor(const double* const* in, double* const* out, int nel, const double* A, long long a_stride,
                               int n_in, int n_out, int S, long long O, const int* shift, void* scratch, int* err,
                               cudaStream_t st);

// One weighted product X^T diag(w v) Y over n points (v may be null): J1 <= 128
// columns of X, J2 of Y; chunks of `chunk` points (gram_tensor_chunk), partial
// c at partial + part + c J1 J2; exponents of its J1 + J2 columns from exp0.
struct TGramTask {
  const double *X, *Y, *w, *v;
  long long part;
  int n, ldx, ldy, J1, J2, chunk, exp0;
  int sym;  // Y = X, J1 = J2 <= 64 in the whole launch, v null and w the square roots of the weights
};
int gram_tensor_chunk(long long n);
// (task, chunk, column chunk) triples
void gram_tensor_items(const TGramTask* tasks, int ntask, std::vector<int>& items);
cudaError_t launch_gram_tensor(const TGramTask* d_tasks, int ntask, const int* d_items, int nitems, int maxJ1, int maxJ2,
                               int* d_exps, double* partial, int* err, cudaStream_t st);

}  // namespace dgdft
