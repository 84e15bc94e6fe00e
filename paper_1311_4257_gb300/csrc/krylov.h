// Vector kernels of the GMRES driver (krylov.cu): complex64 vectors of N values.
#pragma once
#include <cstdint>

#include "common.h"

namespace dfmm {

// Bytes of scratch for vectors of N values and up to ncols basis vectors (zero it once before use).
int64_t krylov_scratch_bytes(int64_t N, int ncols);

// The status word of the apply that a kernel reads the result of, and where the solve gathers them: the
// next apply clears its word.
struct StatusGather {
  const unsigned* word = nullptr;
  unsigned* sum = nullptr;
};

// out = a x + b y (+ c z, where z is given); x, y, z may alias out.
void krylov_combine(float2 a, const float2* x, float2 b, const float2* y, float2 c, const float2* z, float2* out,
                    StatusGather st, int64_t N, cudaStream_t s);

// h[c] = V[c]^H w for c < ncols (V: ncols vectors of N, one after the other).  With u, w is
// first set to a v + b u.
void krylov_dots(const float2* V, int ncols, float2* w, const float2* u, float2 b, const float2* v, float2 a,
                 float2* h, void* scratch, StatusGather st, int64_t N, cudaStream_t s);

// w -= sum_c h[c] V[c]; *norm = |w|.
void krylov_update(const float2* V, int ncols, const float2* h, float2* w, double* norm, void* scratch, int64_t N,
                   cudaStream_t s);

// w /= *norm (nothing where *norm is 0)
void krylov_scale(float2* w, const double* norm, int64_t N, cudaStream_t s);

}  // namespace dfmm
