// Single contractions of the solver as C functions, for the tests of their
// kernels.  Not part of the library's interface (include/bdg.h).
#include <algorithm>

#include "blas.cuh"

namespace bdg {
namespace {

// workspace of one call on its stream
struct Scratch {
  void* p = nullptr;
  cudaStream_t s;
  cudaError_t e;
  Scratch(size_t bytes, cudaStream_t st) : s(st) { e = cudaMallocAsync(&p, bytes, st); }
  ~Scratch() {
    if (p) cudaFreeAsync(p, s);
  }
};

template <typename R>
cudaError_t gram(int digits, const void* A, long long lda, int P, const void* B, long long ldb, int Q, long long n,
                 double* G, cudaStream_t s) {
  typedef typename CT<R>::T T;
  PairBlock<R> a{(const T*)A, lda, n, P}, b{(const T*)B, ldb, n, Q};
  size_t bytes = std::max(gram_workspace_bytes(P, Q, n), gram_digits_workspace_bytes(P, Q, n));
  if (digits == -7) bytes = gram_checked_workspace_bytes(P, Q, n);
  Scratch ws(bytes, s);
  if (ws.e != cudaSuccess) return ws.e;
  if (digits == 0) return gram_pairs<R>(a, b, G, ws.p, bytes, s, false);
  if constexpr (sizeof(R) == 8)
    if (digits == -7) return gram_pairs_checked(a, b, G, ws.p, bytes, s);
  return gram_pairs_digits<R>(a, b, digits, G, ws.p, bytes, s);
}

}  // namespace
}  // namespace bdg

using namespace bdg;

// G as in bdg_gram; digits: 4 or (FP64) 7 by integer digits, -7 by seven with the
// check, 0 on the CUDA cores.  fp64: A and B hold double2, else float2.  Returns a cudaError_t.
extern "C" int bdg_kernel_gram(int fp64, int digits, const void* A, long long lda, int P, const void* B, long long ldb,
                               int Q, long long n, double* G, void* stream) {
  if (!A || !B || !G || P <= 0 || Q <= 0 || n <= 0 || !(digits == 0 || digits == 4 || ((digits == 7 || digits == -7) && fp64)))
    return (int)cudaErrorInvalidValue;
  cudaStream_t s = (cudaStream_t)stream;
  return (int)(fp64 ? gram<double>(digits, A, lda, P, B, ldb, Q, n, G, s) : gram<float>(digits, A, lda, P, B, ldb, Q, n, G, s));
}

// Y = beta Y + alpha A C by integer digits: A P pair columns (double2, lda)
// and Y Q (ldy) of n rows, C 2P x 2Q on the device.  Returns a cudaError_t.
extern "C" int bdg_kernel_update(const void* A, long long lda, int P, const double* C, double beta, double alpha, void* Y,
                                 long long ldy, int Q, long long n, void* stream) {
  if (!A || !C || !Y || P <= 0 || Q <= 0 || n <= 0) return (int)cudaErrorInvalidValue;
  cudaStream_t s = (cudaStream_t)stream;
  Scratch ws(update_digits_workspace_bytes(), s);
  if (ws.e != cudaSuccess) return (int)ws.e;
  return (int)update_pairs_digits(PairBlock<double>{(const double2*)A, lda, n, P}, C, 2 * Q, beta, (double2*)Y, ldy, Q, ws.p, s,
                                  alpha);
}
