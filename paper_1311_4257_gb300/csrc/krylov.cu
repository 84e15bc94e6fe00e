// Vector kernels of the GMRES driver (krylov.h).
//
// They read each basis vector once per pass and are bound by that for large N, by
// launches for small: one pass of classical Gram-Schmidt is two kernels, the
// sums over the blocks are finished by the last block to arrive, and the host
// reads one column of the Hessenberg matrix per iteration (through the vendor library it was
// eight kernels, three waits per iteration and a handle per solve: GMRES on the
// sphere of 4 wavelengths, 16 iterations, 4.6 -> 3.2 ms).  A thread's
// products add in FP32 over at most 4 rows and 32 lanes, the rest in FP64.
#include "krylov.h"

#include "pdl.h"

namespace dfmm {

namespace {

constexpr int KV_T = 256, KV_ROWS = 4, KV_BLOCK = KV_T * KV_ROWS;   // rows per thread, per block
constexpr int KV_GROUP = 64;                                        // columns per shared-memory pass

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ void cfma(float2& c, float2 a, float2 b) {
  c.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x));
  c.y = fmaf(a.x, b.y, fmaf(a.y, b.x, c.y));
}

// whether this block is the last of the grid to get here; its threads then see every block's
// partial sums, and the counter is ready for the next launch
__device__ __forceinline__ bool last_block(unsigned* counter) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
    if (last) *counter = 0u;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

__device__ __forceinline__ void gather(StatusGather st) {
  if (blockIdx.x == 0 && threadIdx.x == 0 && st.word) *st.sum |= *st.word;
}

__global__ __launch_bounds__(KV_T) void combine_kernel(float2 a, const float2* x, float2 b, const float2* y, float2 c,
                                                       const float2* z, float2* out, StatusGather st, int64_t N) {
  pdl_begin();
  gather(st);
  const int64_t i = (int64_t)blockIdx.x * KV_T + threadIdx.x;
  if (i >= N) return;
  float2 r = cmul(a, x[i]);
  cfma(r, b, y[i]);
  if (z) cfma(r, c, z[i]);
  out[i] = r;
}

__global__ __launch_bounds__(KV_T) void dots_kernel(const float2* V, int ncols, float2* w, const float2* u, float2 b,
                                                    const float2* v, float2 a, float2* h, double2* part,
                                                    unsigned* counter, StatusGather st, int64_t N) {
  __shared__ float2 sums[KV_GROUP][KV_T / 32];
  pdl_begin();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t i0 = (int64_t)blockIdx.x * KV_BLOCK + threadIdx.x;
  float2 wv[KV_ROWS];
#pragma unroll
  for (int r = 0; r < KV_ROWS; ++r) {
    const int64_t i = i0 + r * KV_T;
    wv[r] = make_float2(0.f, 0.f);
    if (i < N) {
      if (u) {
        wv[r] = cmul(a, v[i]);
        cfma(wv[r], b, u[i]);
        w[i] = wv[r];
      } else {
        wv[r] = w[i];
      }
    }
  }
  for (int c0 = 0; c0 < ncols; c0 += KV_GROUP) {
    const int nc = min(KV_GROUP, ncols - c0);
    __syncthreads();
#pragma unroll 2
    for (int c = 0; c < nc; ++c) {
      const float2* vc = V + (int64_t)(c0 + c) * N;
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll
      for (int r = 0; r < KV_ROWS; ++r) {
        const int64_t i = i0 + r * KV_T;
        if (i < N) {
          const float2 x = vc[i];
          cfma(acc, make_float2(x.x, -x.y), wv[r]);
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
      }
      if (lane == 0) sums[c][warp] = acc;
    }
    __syncthreads();
    if (threadIdx.x < nc) {
      double2 t = make_double2(0.0, 0.0);
      for (int k = 0; k < KV_T / 32; ++k) {
        t.x += sums[threadIdx.x][k].x;
        t.y += sums[threadIdx.x][k].y;
      }
      part[(int64_t)(c0 + threadIdx.x) * gridDim.x + blockIdx.x] = t;
    }
  }
  gather(st);
  if (!last_block(counter)) return;
  for (int c = warp; c < ncols; c += KV_T / 32) {
    double2 t = make_double2(0.0, 0.0);
    for (unsigned k = lane; k < gridDim.x; k += 32) {
      const double2 p = part[(int64_t)c * gridDim.x + k];
      t.x += p.x;
      t.y += p.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      t.x += __shfl_xor_sync(0xffffffffu, t.x, o);
      t.y += __shfl_xor_sync(0xffffffffu, t.y, o);
    }
    if (lane == 0) h[c] = make_float2((float)t.x, (float)t.y);
  }
}

__global__ __launch_bounds__(KV_T) void update_kernel(const float2* V, int ncols, const float2* h, float2* w,
                                                      double* norm, double2* part, unsigned* counter, int64_t N) {
  __shared__ double sums[KV_T / 32];
  pdl_begin();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t i0 = (int64_t)blockIdx.x * KV_BLOCK + threadIdx.x;
  float2 wv[KV_ROWS];
#pragma unroll
  for (int r = 0; r < KV_ROWS; ++r) wv[r] = i0 + r * KV_T < N ? w[i0 + r * KV_T] : make_float2(0.f, 0.f);
  // the last columns, whose coefficients are small, first, eight at a time: few roundings at the
  // size of w
  for (int c1 = ncols; c1 > 0; c1 -= 8) {
    float2 t[KV_ROWS];
#pragma unroll
    for (int r = 0; r < KV_ROWS; ++r) t[r] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int c = c1 - 1; c >= max(0, c1 - 8); --c) {
      const float2 hc = h[c];
      const float2* vc = V + (int64_t)c * N;
#pragma unroll
      for (int r = 0; r < KV_ROWS; ++r)
        if (i0 + r * KV_T < N) cfma(t[r], hc, vc[i0 + r * KV_T]);
    }
#pragma unroll
    for (int r = 0; r < KV_ROWS; ++r) wv[r] = make_float2(wv[r].x - t[r].x, wv[r].y - t[r].y);
  }
  float n2 = 0.f;
#pragma unroll
  for (int r = 0; r < KV_ROWS; ++r) {
    if (ncols && i0 + r * KV_T < N) w[i0 + r * KV_T] = wv[r];
    n2 = fmaf(wv[r].x, wv[r].x, fmaf(wv[r].y, wv[r].y, n2));
  }
  double t = n2;
  // Where the entries are far from one (about 1e-15, 1e18) their squares leave FP32's range or its full
  // precision; FP64 holds the square of any FP32 number.  Zeros, infinities and NaN come out as themselves.
  if (!(n2 > 1e-30f && n2 < 1e37f)) {
    t = 0.0;
#pragma unroll
    for (int r = 0; r < KV_ROWS; ++r) t += (double)wv[r].x * wv[r].x + (double)wv[r].y * wv[r].y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) sums[warp] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    t = 0.0;
    for (int k = 0; k < KV_T / 32; ++k) t += sums[k];
    part[blockIdx.x].x = t;
  }
  if (!last_block(counter)) return;
  if (warp == 0) {
    t = 0.0;
    for (unsigned k = lane; k < gridDim.x; k += 32) t += part[k].x;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) *norm = sqrt(t);
  }
}

__global__ __launch_bounds__(KV_T) void scale_kernel(float2* w, const double* norm, int64_t N) {
  pdl_begin();
  const int64_t i = (int64_t)blockIdx.x * KV_T + threadIdx.x;
  const double n = *norm;
  if (i >= N || !(n > 0.0)) return;
  const float2 x = w[i];
  if (n > 1e-37 && n < 1e37) {
    const float f = (float)(1.0 / n);
    w[i] = make_float2(x.x * f, x.y * f);
  } else {   // 1 / n is no normal FP32 number
    const double f = 1.0 / n;
    w[i] = make_float2((float)(x.x * f), (float)(x.y * f));
  }
}

int64_t blocks_of(int64_t N) { return (N + KV_BLOCK - 1) / KV_BLOCK; }

// scratch: the arrival counter, then the blocks' partial sums
double2* partials(void* scratch) { return (double2*)((char*)scratch + 256); }

}  // namespace

int64_t krylov_scratch_bytes(int64_t N, int ncols) { return 256 + blocks_of(N) * (ncols > 0 ? ncols : 1) * (int64_t)sizeof(double2); }

void krylov_combine(float2 a, const float2* x, float2 b, const float2* y, float2 c, const float2* z, float2* out,
                    StatusGather st, int64_t N, cudaStream_t s) {
  launch_pdl(combine_kernel, (unsigned)((N + KV_T - 1) / KV_T), KV_T, 0, LaunchStream(s, true), a, x, b, y, c, z, out,
             st, N);
}

void krylov_dots(const float2* V, int ncols, float2* w, const float2* u, float2 b, const float2* v, float2 a,
                 float2* h, void* scratch, StatusGather st, int64_t N, cudaStream_t s) {
  launch_pdl(dots_kernel, (unsigned)blocks_of(N), KV_T, 0, LaunchStream(s, true), V, ncols, w, u, b, v, a, h,
             partials(scratch), (unsigned*)scratch, st, N);
}

void krylov_update(const float2* V, int ncols, const float2* h, float2* w, double* norm, void* scratch, int64_t N,
                   cudaStream_t s) {
  launch_pdl(update_kernel, (unsigned)blocks_of(N), KV_T, 0, LaunchStream(s, true), V, ncols, h, w, norm,
             partials(scratch), (unsigned*)scratch, N);
}

void krylov_scale(float2* w, const double* norm, int64_t N, cudaStream_t s) {
  launch_pdl(scale_kernel, (unsigned)((N + KV_T - 1) / KV_T), KV_T, 0, LaunchStream(s, true), w, norm, N);
}

}  // namespace dfmm
