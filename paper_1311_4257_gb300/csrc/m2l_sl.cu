// Sliced tensor-core form of the translation stage y[dst] += T_op x[src] for the
// tolerances below 1e-5, where the two-term split of m2l_cx.cu is too coarse:
// products of FP32 or FP64 accuracy on the FP16 tensor cores.
//
// A state's entries span many decades, and so do an operator's columns and rows: what its
// representation resolves least is what a touching-shell operator amplifies most (eps
// 1e-8, boxes of half a wavelength: states 2.6e2 to 1e-6, columns 0.6 to 80).  Powers of two
// even them out first, exactly: c_q per entry of a state, the largest |T[p][q]| of all the
// operators that read it, at most 1; d_p per row of an operator, above its |T[p][q]| / c_q; and
// s per gathered row, above its c_q |x_q|.  The scaled values (|v| <= 1) are
// cut into S FP16 slices v = sum_i v_i B^-i.  The product keeps the slice pairs
// i + j < S; the pairs of one sum g = i + j share the weight B^-g and accumulate
// in one tensor-memory accumulator ("group" g) of the FP32-accumulating MMA.
//
//  * FP32 rows, S = 3, B = 2^8: v_0 is an 8-bit integer (128 v rounded), v_1 and
//    v_2 are FP16 numbers that hold the rest to 2^-20 and 2^-31 of the row's
//    largest entry.  Group 0 sums integers below 2 K 2^14 <= 2^24 (K <= 512): it is
//    exact.  The accumulators of groups 1 and 2 truncate at 2^-24 of terms that
//    weigh 2^-8 and 2^-16, and the dropped pairs weigh 2^-27.
//  * FP64 rows, S = 8, B = 2^7: v = sum_i d_i 2^-(6 + 7 i) with balanced 7-bit
//    integers |d_i| <= 64, to 2^-56 of the row's largest entry.  Group g
//    sums (g + 1) 2 K products of at most 2^12, below 2^24 and so exact for
//    (g + 1) K <= 2048; K <= 512 covers groups 0 to 3, and a truncation in group 4
//    or later weighs 2^-24 2^-28 at most.  The epilogue joins the eight integers in
//    64-bit arithmetic, to 2^-52, and rounds to FP64.
//
// So the error is fixed against the largest possible product, not against each: what one stage
// loses depends on how even the scaled values are.  Emulated on operators and states of the
// representations (boxes of 1/2 and 1/4, offsets from touching to far and M2M; relative 2-norm
// against 80-bit products): FP32 4e-8 to 1e-7, where an FP32 FMA chain makes 3e-7 to
// 1e-6; FP64 4e-16 to 3e-15, where an FP64 chain makes 4e-16 to 2e-15.  With one power of two per
// operator and per row it was 8e-8 to 8e-7 and 5e-15 to 6e-13.
//
// One CTA computes 128 gathered columns (pairs x right-hand sides) against a
// block of n outputs (n <= 80, 32): operator slices of the block are stacked as
// rows of the MMA's B operand, so one MMA of N = (S - i) n multiplies slice i of
// the columns by operator slices 0 .. S - 1 - i and lands on the groups
// i .. S - 1, which are adjacent tensor-memory columns.  An MMA of M = 128, K = 16
// takes max(N / 2, 32 + N / 4) clocks (the second: its operands at 128 bytes per
// clock of shared memory), so stacked N of 64 to 256 run at 62 to 100% of the
// rate where N = 32 would run at 40%.
//
// A chunk is 64 K values, so that a row's piece of one slice is one 128-byte line
// in global memory and one swizzled row in shared memory: cp.async takes a
// shared-memory pass per global line an instruction touches (16-value chunks,
// 16 lines per instruction: 19 passes instead of 4; 4.16 -> 3.76 ms on the case below).
//
// The MMA warp issues converged, from an elected lane (tcgen05.cuh); from one diverged
// thread the issue of an MMA, 115 to 140 clocks, was the longest part of an item (16.7k
// clocks, 10k at the MMAs' own rate).
//
// Measured against the CUDA-core stages that served these tolerances: sphere of 32
// wavelengths, eps 1e-6 (N = 321,699, FP32): all translations 19.2 -> 2.55 ms, 22
// -> 168 TFLOP/s (of 327 at the MMAs' rate); sphere of 8, eps 1e-8 (FP64): 68 ->
// 2.41 ms, 0.75 -> 21 TFLOP/s.  The warp-wide issue gave the applies 3.76 -> 2.88 and
// 3.78 -> 3.03 ms of that.  It is bound by shared-memory bandwidth (operand reads and
// the copies into the tiles) where tiles are full, by part-filled tiles elsewhere.
#include <cuda_fp16.h>

#include <algorithm>

#include "apply.h"
#include "pdl.h"
#include "per_device.h"
#include "tcgen05.cuh"

namespace dfmm {

namespace {

using namespace tc;

constexpr int SL_M = 128;            // gathered columns per tile
constexpr int SL_K = 64;             // K values per chunk: a 128-byte line, four MMA steps
constexpr int SL_ROW = 128;          // bytes of one slice of one row's chunk
constexpr int SL_TILE = SL_M * SL_ROW;   // 16 KB: one slice of the gathered chunk
constexpr int SL_PRODUCERS = 128;    // warps 0-3: gather; 4-11: epilogue; 12: MMA issuer
constexpr int SL_MMA_WARP = 12;
constexpr int SL_THREADS = 416;
constexpr int SL_TMEM_COLS = 512;
constexpr int SL_KMAX = 512;         // exactness of the integer groups (file comment)

// S slices; n outputs per block (2 S n <= 512 tensor-memory columns); slots of the
// two shared-memory rings: 16 KB tiles of gathered columns, and chunks of operator slices
template <int S> struct Cfg;
template <> struct Cfg<3> { static constexpr int N = 80, NA = 6, NB = 2; };
template <> struct Cfg<8> { static constexpr int N = 32, NA = 6, NB = 2; };

template <int S> __host__ __device__ constexpr int b_bytes_max() { return 2 * S * Cfg<S>::N * SL_ROW; }
template <int S> constexpr int sl_smem() { return Cfg<S>::NA * SL_TILE + Cfg<S>::NB * b_bytes_max<S>() + 1024 + 512; }
static_assert(sl_smem<3>() <= 232448 - 1024 && sl_smem<8>() <= 232448 - 1024, "shared memory per CTA");
static_assert(2 * 3 * Cfg<3>::N <= SL_TMEM_COLS && 2 * 8 * Cfg<8>::N <= SL_TMEM_COLS, "tensor memory");

__host__ __device__ __forceinline__ int round16(int x) { return (x + 15) & ~15; }

// outputs per block for target rank M: blocks of equal size, a multiple of 16
template <int S> __host__ __device__ __forceinline__ int block_rows(int M) {
  const int nb = (M + Cfg<S>::N - 1) / Cfg<S>::N;
  return round16((M + nb - 1) / nb);
}

// ---------------------------------------------------------------- slices ---

// scale 2^e >= |m| from the largest magnitude's bits; NaN or infinity anywhere in the row
// gives a NaN scale (its digits are zero), so the products are NaN as well
__device__ __forceinline__ void scale32(uint32_t mbits, float& s, float& inv) {
  if (mbits >= 0x7f800000u) { s = __uint_as_float(0x7fc00000u); inv = 0.f; return; }
  uint32_t e = (mbits + 0x7fffffu) >> 23;         // exponent of the power of two >= m
  e = min(max(e, 1u), 253u);                      // 2^-126 .. 2^126: s and 1 / s stay normal
  s = __uint_as_float(e << 23);
  inv = __uint_as_float((254u - e) << 23);
}
__device__ __forceinline__ void scale64(uint32_t mhi, double& s, double& inv) {
  if (mhi >= 0x7ff00000u) { s = __hiloint2double(0x7ff80000, 0); inv = 0.0; return; }
  uint32_t e = (mhi >> 20) + 1u;                  // 2^e > m
  e = min(max(e, 1u), 2045u);
  s = __hiloint2double((int)(e << 20), 0);
  inv = __hiloint2double((int)((2046u - e) << 20), 0);
}

__device__ __forceinline__ void slice(float v, __half (&d)[3]) {
  const float t = v * 128.f;
  const float d0 = rintf(t);
  const float r = (t - d0) * 256.f;               // |r| <= 128, exact
  const __half h1 = __float2half_rn(r);
  d[0] = __float2half_rn(d0);
  d[1] = h1;
  d[2] = __float2half_rn((r - __half2float(h1)) * 256.f);
}
__device__ __forceinline__ void slice(double v, __half (&d)[8]) {
  constexpr long long kBias = 64ll * (1ll + (1ll << 7) + (1ll << 14) + (1ll << 21) + (1ll << 28) + (1ll << 35) + (1ll << 42));
  const unsigned long long I = (unsigned long long)(__double2ll_rn(v * 36028797018963968.0) + kBias);   // 2^55 v
#pragma unroll
  for (int i = 0; i < 7; ++i) d[7 - i] = __int2half_rn((int)((I >> (7 * i)) & 127u) - 64);
  d[0] = __int2half_rn((int)((long long)I >> 49));
}

// 8 consecutive values of one slice as one 16-byte piece
template <int S>
__device__ __forceinline__ void store_pieces(unsigned char* out, const __half (*d)[S]) {
#pragma unroll
  for (int i = 0; i < S; ++i) {
    uint4 w;
    __half2 p[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) p[k] = __halves2half2(d[2 * k][i], d[2 * k + 1][i]);
    w = *(uint4*)p;
    *(uint4*)(out + i * SL_ROW) = w;
  }
}

// the largest of the magnitudes of a value's parts, as bits that compare like it (of a double its high word)
__device__ __forceinline__ uint32_t mag_bits(float2 v) {
  return max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu);
}
__device__ __forceinline__ uint32_t mag_bits(double2 v) {
  return max((uint32_t)__double2hiint(v.x) & 0x7fffffffu, (uint32_t)__double2hiint(v.y) & 0x7fffffffu);
}
template <class T2, class T> __device__ __forceinline__ T2 scaled(T2 v, T f) { return T2{v.x * f, v.y * f}; }

// 8 consecutive values of a row, times their scales
__device__ __forceinline__ void load_piece(const float2* x, const float* col, float2 (&v)[8]) {
  const float4 c0 = ((const float4*)col)[0], c1 = ((const float4*)col)[1];
  const float c[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float4 w = ((const float4*)x)[k];
    v[2 * k] = make_float2(w.x * c[2 * k], w.y * c[2 * k]);
    v[2 * k + 1] = make_float2(w.z * c[2 * k + 1], w.w * c[2 * k + 1]);
  }
}
__device__ __forceinline__ void load_piece(const double2* x, const double* col, double2 (&v)[8]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double2 c = ((const double2*)col)[k];
    v[2 * k] = scaled(x[2 * k], c.x);
    v[2 * k + 1] = scaled(x[2 * k + 1], c.y);
  }
}

// Source rows (r complex values each, r a multiple of 8), times col[q] -> slices [row][chunk][re, im][slice][64]
// (r to a multiple of 16 with zeros; what is left of the last chunk is not read), one scale per row.  One warp per row;
// a lane takes 8 complex values, i.e. one 16-byte piece of every slice, and holds those of its first
// piece (all of them up to rank 256) while the row's largest entry is found.
template <int S, class T2, class T>
__global__ __launch_bounds__(256) void split_sl_kernel(const T2* x, const T* col, int64_t rows, int r, unsigned char* out,
                                                       T* scale) {
  pdl_begin();
  const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  const T2* xr = x + row * r;
  const int nx = r / 8, np = round16(r) / 8;   // pieces with values, pieces
  T2 v[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = T2{T(0), T(0)};
  uint32_t m = 0;
  if (lane < nx) load_piece(xr + 8 * lane, col + 8 * lane, v);
#pragma unroll
  for (int k = 0; k < 8; ++k) m = max(m, mag_bits(v[k]));
  for (int q = lane + 256; q < r; q += 32) m = max(m, mag_bits(scaled(xr[q], col[q])));
  m = __reduce_max_sync(0xffffffffu, m);
  T s, inv;
  if constexpr (S == 3) scale32(m, s, inv);
  else scale64(m, s, inv);
  if (lane == 0) scale[row] = s;
  const bool fin = s == s;
  unsigned char* o = out + row * (int64_t)((r + SL_K - 1) / SL_K * 2 * S * SL_ROW);
  for (int p = lane; p < np; p += 32) {
    if (p >= 32 && p < nx) load_piece(xr + 8 * p, col + 8 * p, v);
    if (!fin || p >= nx)
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = T2{T(0), T(0)};
    __half d[8][S];
    unsigned char* oc = o + (p >> 3) * (2 * S * SL_ROW) + (p & 7) * 16;
#pragma unroll
    for (int k = 0; k < 8; ++k) slice(v[k].x * inv, d[k]);
    store_pieces<S>(oc, d);
#pragma unroll
    for (int k = 0; k < 8; ++k) slice(v[k].y * inv, d[k]);
    store_pieces<S>(oc + S * SL_ROW, d);
  }
}

// bits[q] = max of mag_bits over the entries of column q of all operators; one block per operator
template <class T2>
__global__ __launch_bounds__(256) void op_col_max_kernel(const T2* __restrict__ ops, int M, int Kd, uint32_t* bits) {
  const T2* a = ops + (int64_t)blockIdx.x * M * Kd;
  for (int q = threadIdx.x; q < Kd; q += 256) {
    uint32_t m = 0;
    for (int p = 0; p < M; ++p) m = max(m, mag_bits(a[(int64_t)p * Kd + q]));
    atomicMax(bits + q, m);
  }
}

// col[q] = the power of two of column q over that of the largest column, at least 2^-100, and 1 where
// nothing reads the entry (padding); one block
template <class T, int MANT>
__global__ __launch_bounds__(512) void op_col_scale_kernel(const uint32_t* __restrict__ bits, int Kd, T* __restrict__ col) {
  __shared__ int top;
  if (threadIdx.x == 0) top = 0;
  __syncthreads();
  const int q = threadIdx.x, e = q < Kd ? (int)(bits[q] >> MANT) : 0;
  atomicMax(&top, e);
  __syncthreads();
  if (q < Kd) col[q] = bits[q] == 0 ? T(1) : (T)__uint_as_float((uint32_t)(127 + max(e - top, -100)) << 23);
}

// row[op][p] (rows of Mp values): a power of two above |T[p][q]| / col[q] for every q, times the unit
// that the groups are joined in; a warp per row
template <class T> __host__ __device__ constexpr T sl_unit() { return sizeof(T) == 4 ? T(6.103515625e-05) : T(2.220446049250313e-16); }   // 2^-14, 2^-52

template <class T2, class T>
__global__ __launch_bounds__(256) void op_row_scale_kernel(const T2* __restrict__ ops, const T* __restrict__ col, int M,
                                                           int Kd, int Mp, int64_t rows, T* __restrict__ row) {
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= rows) return;
  const T2* a = ops + i * Kd;
  uint32_t m = 0;
  for (int q = lane; q < Kd; q += 32) m = max(m, mag_bits(scaled(a[q], T(1) / col[q])));
  m = __reduce_max_sync(0xffffffffu, m);
  T s, inv;
  if constexpr (sizeof(T) == 4) scale32(m, s, inv);
  else scale64(m, s, inv);
  if (lane == 0) row[i / M * Mp + i % M] = s * sl_unit<T>();
}

// Operator image [op][block][chunk][Tr, Ti][slice][row of the block][64], zero beyond M
// and Kd, each row of 128 bytes swizzled as the MMA reads it: a chunk is one
// bulk copy and the slices of Tr (or Ti) are one stacked operand.  One block per (op, chunk).
template <int S, class T2, class T>
__global__ __launch_bounds__(256) void op_image_sl_kernel(const T2* __restrict__ ops, const T* __restrict__ col,
                                                          const T* __restrict__ rows, int M, int Kd,
                                                          unsigned char* __restrict__ img) {
  const int nchunk = (Kd + SL_K - 1) / SL_K, Mp = round16(M), n = block_rows<S>(M);
  const int64_t op = blockIdx.x / nchunk;
  const int c = (int)(blockIdx.x % nchunk);
  const T2* top = ops + op * (int64_t)M * Kd;
  unsigned char* base = img + op * (int64_t)nchunk * 2 * S * SL_ROW * Mp;
  for (int e = threadIdx.x; e < Mp * 8; e += blockDim.x) {
    const int p = e >> 3, pc = e & 7;
    const int blk = p / n, row = p - blk * n, nb = min(n, Mp - blk * n);
    unsigned char* o = base + (int64_t)blk * n * (nchunk * 2 * S * SL_ROW) + (int64_t)c * (2 * S * SL_ROW * nb);
    const T inv = p < M ? sl_unit<T>() / rows[op * Mp + p] : T(0);
    T2 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int q = c * SL_K + 8 * pc + k;
      v[k] = T2{T(0), T(0)};
      if (p < M && q < Kd) v[k] = scaled(scaled(top[(int64_t)p * Kd + q], T(1) / col[q]), inv);
    }
#pragma unroll
    for (int part = 0; part < 2; ++part) {
      __half d[8][S];
#pragma unroll
      for (int k = 0; k < 8; ++k) slice(part ? v[k].y : v[k].x, d[k]);
#pragma unroll
      for (int i = 0; i < S; ++i) {
        __half2 w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = __halves2half2(d[2 * k][i], d[2 * k + 1][i]);
        *(uint4*)(o + (part * S + i) * (SL_ROW * nb) + sw128_off(row, pc)) = *(uint4*)w;
      }
    }
  }
}

// --------------------------------------------------------------- kernel ----

// 16 lanes x 8 columns (.16x256b): thread t gets lane t / 4 (r[0], r[1]) and lane
// t / 4 + 8 (r[2], r[3]) at columns 2 (t % 4) + {0, 1}
__device__ __forceinline__ void tmem_ld16x256_x1(uint32_t ta, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(ta));
}

__device__ __forceinline__ void red_add_f64(double* p, double v) {
  asm volatile("red.relaxed.gpu.global.add.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

// The groups of one output, r[4 g] the group's accumulator, as the stage's value / (row scale x column scale).
__device__ __forceinline__ float join3(const uint32_t* r) {
  return __uint_as_float(r[0]) + (__uint_as_float(r[4]) + __uint_as_float(r[8]) * 0.00390625f) * 0.00390625f;
}
// |sum| <= 2 K <= 2^10, in units of 2^-52, so the 64-bit integer does not overflow
__device__ __forceinline__ double join8(const uint32_t* r) {
  int s[8];
#pragma unroll
  for (int g = 0; g < 8; ++g) s[g] = __float2int_rn(__uint_as_float(r[4 * g]));
  long long hi = s[0], lo = s[4];
#pragma unroll
  for (int g = 1; g < 4; ++g) {
    hi = hi * 128 + s[g];
    lo = lo * 128 + s[4 + g];
  }
  return (double)(hi * (1 << 19) + ((lo + 256) >> 9));
}

// Persistent, warp-specialised; item = (tile, block of n outputs), CTA x takes
// items x, x + gridDim.x, ..., so the CTAs that run together share a tile's
// gathered rows in L2.
//   warps 0-3  producers: 8 lanes copy one row of a tile (a slice of the real or
//              imaginary parts, one 128-byte line) with 16-byte cp.async into the
//              swizzled tile; thread 0 also bulk-copies the operator chunk.
//   warp 12    an elected lane issues the two stacked MMAs of every K step of a tile.
//   warps 4-11 epilogue: join the groups of an output into registers, hand the
//              accumulators back, scale, add to the target row.
// Every wait is time-limited; on a timeout the CTA reports it, stops issuing,
// lets its own copies and MMAs land, frees its tensor memory and returns.
template <int S, class T2, class T>
__global__ __launch_bounds__(SL_THREADS, 1) void gemm_sl_kernel(GemmArgs a, SlArgs t, int nblk, unsigned* status) {
  pdl_begin();
  constexpr int NA = Cfg<S>::NA, NB = Cfg<S>::NB;
  constexpr int RPT = SL_M * 8 / SL_PRODUCERS;   // rows per producer thread
  extern __shared__ unsigned char smem_raw[];
  __shared__ int s_start;
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t sA = smem_u32(smem), sB = sA + NA * SL_TILE;
  uint64_t* fullA = (uint64_t*)(smem + NA * SL_TILE + NB * b_bytes_max<S>());
  uint64_t* emptyA = fullA + NA;
  uint64_t* fullB = emptyA + NA;
  uint64_t* emptyB = fullB + NB;
  uint64_t* acc_full = emptyB + NB;
  uint64_t* acc_empty = acc_full + 1;
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int M = a.M, Mp = round16(M), n = block_rows<S>(M);
  const int nchunk = (a.Kd + SL_K - 1) / SL_K;
  const int nitems = (int)a.ntiles * nblk, G = (int)gridDim.x;
  const int64_t row_bytes = (int64_t)nchunk * 2 * S * SL_ROW;   // of a source row, and of an operator row

  if (tid == 0) s_start = (*(volatile unsigned*)status & kStatusTimeout) ? 0 : 1;
  __syncthreads();
  if (!s_start) return;   // an earlier CTA gave up: skip the work, hold no tensor memory
  if (tid == 0) {
    for (int i = 0; i < NA; ++i) {
      mbar_init(smem_u32(&fullA[i]), SL_PRODUCERS);
      mbar_init(smem_u32(&emptyA[i]), 1);
    }
    for (int i = 0; i < NB; ++i) {
      mbar_init(smem_u32(&fullB[i]), 1);
      mbar_init(smem_u32(&emptyB[i]), 1);
    }
    mbar_init(smem_u32(acc_full), 1);
    mbar_init(smem_u32(acc_empty), 8);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == SL_MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(SL_TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp < SL_PRODUCERS / 32) {
    // ---------------- producers ----------------
    const int pc = tid & 7, r0 = tid >> 3;   // 16-byte piece; rows r0 + 16 q
    constexpr int RSTEP = SL_PRODUCERS / 8;
    const unsigned char* src = (const unsigned char*)t.src;
    const uint32_t dst0 = sw128_off(r0, pc);
    const int kp = round16(a.Kd);
    auto load_rows = [&](int4 tl, int* rows) {
      const int ncol = tl.z * a.nrhs;
      const uint32_t mg = rhs_magic(a.nrhs);
#pragma unroll
      for (int q = 0; q < RPT; ++q) {
        const int col = r0 + q * RSTEP;
        rows[q] = -1;
        if (col < ncol) {
          const int pr = div_rhs(col, mg);
          rows[q] = a.pairs[tl.y + pr].x * a.nrhs + (col - pr * a.nrhs);
        }
      }
    };
    // the next item's rows are looked up while this item's chunks are issued
    const int4 none = make_int4(0, 0, 0, 0);
    int it = (int)blockIdx.x;
    int4 tile_n = it < nitems ? a.tiles[it / nblk] : none;
    int rows_n[RPT];
    load_rows(tile_n, rows_n);
    int4 tile_nn = it + G < nitems ? a.tiles[(it + G) / nblk] : none;
    Ring ra, rb;
    int ga = 0, gb = 0;   // slots filled so far (up to the ring's size: no wait on the first round)
    bool ok = true;
    for (; it < nitems && ok; it += G) {
      const unsigned char* srow[RPT];
#pragma unroll
      for (int q = 0; q < RPT; ++q) srow[q] = rows_n[q] >= 0 ? src + rows_n[q] * row_bytes + 16 * pc : nullptr;
      const int blk = it % nblk, nb = min(n, Mp - blk * n);
      const uint32_t bb = (uint32_t)(2 * S * SL_ROW * nb);
      const unsigned char* img = (const unsigned char*)t.img + tile_n.x * (row_bytes * Mp) + blk * n * row_bytes;
      tile_n = tile_nn;
      load_rows(tile_n, rows_n);
      tile_nn = it + 2 * G < nitems ? a.tiles[(it + 2 * G) / nblk] : none;
      for (int c = 0; c < nchunk && ok; ++c) {
        if (warp == 0) {   // operator chunk: Tr slices, Ti slices
          int okw = 1;
          if (lane == 0) {
            if (gb >= NB) okw = mbar_wait(smem_u32(&emptyB[rb.st]), rb.ph ^ 1u, status) ? 1 : 0;
            if (okw) {
              mbar_expect_tx(smem_u32(&fullB[rb.st]), bb);
              bulk_g2s(sB + rb.st * b_bytes_max<S>(), img + c * (int64_t)bb, bb, smem_u32(&fullB[rb.st]));
            }
          }
          ok = __shfl_sync(0xffffffffu, okw, 0) != 0;
          if (!ok) break;
          ++gb;
          rb.next(NB);
        }
        const bool kin = c * SL_K + 8 * pc < kp;
        for (int h = 0; h < 2 * S; ++h) {   // tiles: slices of the real, then of the imaginary parts
          if (ga >= NA) {   // the slot's previous tile has been consumed by the MMAs
            int okw = 0;
            if (lane == 0) okw = mbar_wait(smem_u32(&emptyA[ra.st]), ra.ph ^ 1u, status) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, okw, 0) != 0;
            if (!ok) break;
          }
          const uint32_t d = sA + ra.st * SL_TILE + dst0;
          const int off = (c * 2 * S + h) * SL_ROW;
          if (kin) {
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
              if (srow[q]) cp_async16(d + q * (RSTEP * SL_ROW), srow[q] + off);
              else cp_async16_zero(d + q * (RSTEP * SL_ROW), src);
            }
          }
          asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&fullA[ra.st])) : "memory");
          ga = min(ga + 1, NA);
          ra.next(NA);
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (tid == 0)   // the bulk copies of the last fills have landed
      for (int q = 0; q < min(gb, NB); ++q) {
        const int g = gb - 1 - q;
        mbar_wait_drain(smem_u32(&fullB[g % NB]), (uint32_t)((g / NB) & 1));
      }
  } else if (warp == SL_MMA_WARP) {
    // ---------------- MMA issuer ----------------
    {
      const uint32_t lead = elect_one(), tm = __reduce_max_sync(0xffffffffu, tmem);   // uniform
      Ring ra, rb;
      int last = -1, i = 0;
      uint32_t last_ph = 0;
      const int kp = round16(a.Kd);
      bool ok = true;
      for (int it = (int)blockIdx.x; it < nitems && ok; it += G, ++i) {
        const int blk = it % nblk, nb = min(n, Mp - blk * n);
        if (i > 0 && !warp_wait(smem_u32(acc_empty), (uint32_t)((i - 1) & 1), status)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        for (int c = 0; c < nchunk && ok; ++c) {
          if (!warp_wait(smem_u32(&fullB[rb.st]), rb.ph, status)) {
            ok = false;
            break;
          }
          const int ksteps = min(SL_K, kp - c * SL_K) / 16;
          const uint32_t tr = sB + rb.st * b_bytes_max<S>(), ti = tr + (uint32_t)(S * SL_ROW * nb);
          for (int h = 0; h < 2 * S; ++h) {
            if (!warp_wait(smem_u32(&fullA[ra.st]), ra.ph, status)) {
              ok = false;
              break;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // cp.async data -> async proxy
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // Re y = Tr xr - Ti xi, Im y = Ti xr + Tr xi; slice sl of the columns against slices 0 .. S - 1 - sl
            const bool im = h >= S;
            const int sl = im ? h - S : h;
            const uint32_t xa = sA + ra.st * SL_TILE, b_re = im ? ti : tr, b_im = im ? tr : ti;
            const uint32_t d_re = tm + (uint32_t)(sl * nb), d_im = d_re + (uint32_t)(S * nb);
            const uint32_t id_re = idesc_f16((S - sl) * nb, im), id_im = idesc_f16((S - sl) * nb);
            for (int k = 0; k < ksteps; ++k) {
              const uint64_t da = smem_desc_sw128(xa + 32 * k);
              const uint32_t acc = (c > 0 || h > 0 || k > 0) ? 1u : 0u;   // the first covers every group
              mma_f16_by(lead, d_re, da, smem_desc_sw128(b_re + 32 * k), id_re, acc);
              mma_f16_by(lead, d_im, da, smem_desc_sw128(b_im + 32 * k), id_im, acc);
            }
            mma_commit_by(lead, smem_u32(&emptyA[ra.st]));
            last = ra.st;
            last_ph = ra.ph;
            ra.next(NA);
          }
          if (!ok) break;
          mma_commit_by(lead, smem_u32(&emptyB[rb.st]));
          rb.next(NB);
        }
        if (!ok) break;
        mma_commit_by(lead, smem_u32(acc_full));
      }
      // MMAs complete in order: once the last commit has arrived, all have
      if (last >= 0) mbar_wait_drain(smem_u32(&emptyA[last]), last_ph);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue ----------------
    // warp 4 + w takes tensor-memory lanes 32 (w % 4) .. and every other 8 columns of a group
    const int quarter = warp & 3, par = (warp - SL_PRODUCERS / 32) >> 2;
    constexpr int STEPS = (Cfg<S>::N / 8 + 1) / 2;
    int i = 0;
    for (int it = (int)blockIdx.x; it < nitems; it += G, ++i) {
      const int4 tile = a.tiles[it / nblk];
      const int blk = it % nblk, nb = min(n, Mp - blk * n);
      const int ncol = tile.z * a.nrhs;
      const uint32_t mg = rhs_magic(a.nrhs);
      T* out[4];
      T cs[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {   // columns 32 quarter + 16 (h / 2) + lane / 4 + 8 (h % 2)
        const int col = 32 * quarter + 16 * (h >> 1) + (lane >> 2) + 8 * (h & 1);
        out[h] = nullptr;
        cs[h] = T(0);
        if (col < ncol) {
          const int q = div_rhs(col, mg);
          const int2 pr = a.pairs[tile.y + q];
          const int k = col - q * a.nrhs;
          cs[h] = ((const T*)t.src_scale)[(int64_t)pr.x * a.nrhs + k];
          out[h] = (T*)((T2*)a.dst + ((int64_t)pr.y * a.nrhs + k) * a.dst_ld) + 2 * blk * n + 4 * (lane & 3);
        }
      }
      const int nout = min(nb, M - blk * n);   // outputs of the block; the rest pads it
      // row scales: of this thread's outputs, 8 (2 j + par) + 2 (lane % 4) + {0, 1}, at rs[8 j]; the block's are on
      // their way to L1 while the MMAs run
      const T* rs0 = (const T*)t.row_scale + (int64_t)tile.x * Mp + blk * n;
      const T2* rs = (const T2*)(rs0 + 8 * par + 2 * (lane & 3));
      if (lane * 32 < nb * (int)sizeof(T)) asm volatile("prefetch.global.L1 [%0];" ::"l"((const char*)rs0 + lane * 32));
      int okw = 0;
      if (lane == 0) okw = mbar_wait(smem_u32(acc_full), (uint32_t)(i & 1), status) ? 1 : 0;
      okw = __shfl_sync(0xffffffffu, okw, 0);
      if (!okw) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // join the groups into registers and hand the accumulators back before the additions to global memory
      T y[2][STEPS][2][4];
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const uint32_t tb = tmem + ((uint32_t)(32 * quarter + 16 * b) << 16);
#pragma unroll
        for (int j = 0; j < STEPS; ++j) {
          const int j0 = 8 * (2 * j + par);
          if (j0 < nout) {   // warp-uniform
            uint32_t v[4 * S];
#pragma unroll
            for (int part = 0; part < 2; ++part) {
#pragma unroll
              for (int g = 0; g < S; ++g) tmem_ld16x256_x1(tb + (uint32_t)((part * S + g) * nb + j0), v + 4 * g);
              asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
              for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                  if constexpr (S == 3) y[b][j][h][2 * e + part] = join3(v + 2 * h + e);
                  else y[b][j][h][2 * e + part] = join8(v + 2 * h + e);
                }
            }
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(acc_empty)) : "memory");
      T2 so[STEPS];   // loaded here: the registers were the accumulators' until now
#pragma unroll
      for (int j = 0; j < STEPS; ++j) so[j] = 8 * (2 * j + par) < nout ? rs[8 * j] : T2{T(0), T(0)};
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int j = 0; j < STEPS; ++j) {
          const int j0 = 8 * (2 * j + par);
          if (j0 >= nout) break;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            T* o = out[2 * b + h] + 2 * j0;
            const T* v = y[b][j][h];
            if (out[2 * b + h]) {
              if constexpr (S == 3) {
                const float c = cs[2 * b + h];
                red_add4(o, v[0] * so[j].x * c, v[1] * so[j].x * c, v[2] * so[j].y * c, v[3] * so[j].y * c);
              } else {
                const double c0 = so[j].x * cs[2 * b + h], c1 = so[j].y * cs[2 * b + h];
#pragma unroll
                for (int e = 0; e < 4; ++e) red_add_f64(o + e, v[e] * (e < 2 ? c0 : c1));
              }
            }
          }
        }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == SL_MMA_WARP)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(SL_TMEM_COLS));
}

template <int S, class T2, class T>
void launch_sl(const GemmArgs& a, const SlArgs& t, unsigned* status, LaunchStream s) {
  static PerDevice<int> sms;   // set up with the kernel's launch attribute
  int dev = 0;
  DFMM_CUDA(cudaGetDevice(&dev));
  const int nsm = sms.get(dev, [&] {
    int n = 0;
    DFMM_CUDA(cudaFuncSetAttribute(gemm_sl_kernel<S, T2, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, sl_smem<S>()));
    DFMM_CUDA(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
    return n;
  });
  const int n = block_rows<S>(a.M), nblk = (a.M + n - 1) / n;
  const int64_t items = a.ntiles * nblk;
  if (items > INT32_MAX - 1024) throw Error(-5, "translation stage has too many work items");
  launch_pdl(gemm_sl_kernel<S, T2, T>, (unsigned)std::min<int64_t>(items, nsm), SL_THREADS, sl_smem<S>(), s, a, t, nblk, status);
  DFMM_CUDA(cudaGetLastError());
}

}  // namespace

bool gemm_sl_supported(int M, int Kd) { return M % 8 == 0 && Kd % 8 == 0 && M >= 8 && Kd >= 8 && M <= 512 && Kd <= SL_KMAX; }

int64_t sl_row_bytes(int r, bool fp64) { return (int64_t)((r + SL_K - 1) / SL_K) * 2 * (fp64 ? 8 : 3) * SL_ROW; }

int64_t sl_image_bytes(int M, int Kd, int nops, bool fp64) { return (int64_t)nops * round16(M) * sl_row_bytes(Kd, fp64); }

int sl_padded_rows(int M) { return round16(M); }

void sl_column_max(const void* ops, int M, int Kd, int nops, uint32_t* bits, bool fp64, cudaStream_t s) {
  if (nops == 0) return;
  if (fp64) op_col_max_kernel<<<nops, 256, 0, s>>>((const double2*)ops, M, Kd, bits);
  else op_col_max_kernel<<<nops, 256, 0, s>>>((const float2*)ops, M, Kd, bits);
  DFMM_CUDA(cudaGetLastError());
}

void sl_column_scales(const uint32_t* bits, int Kd, void* col, bool fp64, cudaStream_t s) {
  if (Kd > SL_KMAX) throw Error(-5, "sliced stage needs ranks up to 512");
  if (fp64) op_col_scale_kernel<double, 20><<<1, SL_KMAX, 0, s>>>(bits, Kd, (double*)col);
  else op_col_scale_kernel<float, 23><<<1, SL_KMAX, 0, s>>>(bits, Kd, (float*)col);
  DFMM_CUDA(cudaGetLastError());
}

template <int S, class T2, class T>
void build_sl(const T2* ops, const T* col, int M, int Kd, int nops, unsigned char* img, T* row, cudaStream_t s) {
  const int64_t rows = (int64_t)nops * M;
  op_row_scale_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(ops, col, M, Kd, round16(M), rows, row);
  op_image_sl_kernel<S><<<(unsigned)((int64_t)nops * ((Kd + SL_K - 1) / SL_K)), 256, 0, s>>>(ops, col, row, M, Kd, img);
  DFMM_CUDA(cudaGetLastError());
}

void build_sl_image(const void* ops, const void* col, int M, int Kd, int nops, void* img, void* row, bool fp64,
                    cudaStream_t s) {
  if (nops == 0) return;
  if (!gemm_sl_supported(M, Kd)) throw Error(-5, "sliced stage needs ranks that are multiples of 8, <= 512");
  unsigned char* p = (unsigned char*)img;
  if (fp64) build_sl<8>((const double2*)ops, (const double*)col, M, Kd, nops, p, (double*)row, s);
  else build_sl<3>((const float2*)ops, (const float*)col, M, Kd, nops, p, (float*)row, s);
}

void launch_split_sl(const float2* x, const void* col, int64_t rows, int r, void* out, void* scale, bool fp64,
                     LaunchStream s) {
  if (rows == 0) return;
  const unsigned grid = (unsigned)((rows * 32 + 255) / 256);
  if (fp64)
    launch_pdl(split_sl_kernel<8, double2, double>, grid, 256, 0, s, (const double2*)x, (const double*)col, rows, r,
               (unsigned char*)out, (double*)scale);
  else
    launch_pdl(split_sl_kernel<3, float2, float>, grid, 256, 0, s, x, (const float*)col, rows, r, (unsigned char*)out,
               (float*)scale);
  DFMM_CUDA(cudaGetLastError());
}

void launch_gemm_stage_sl(const GemmArgs& a, const SlArgs& t, unsigned* status, bool fp64, LaunchStream s) {
  if (a.ntiles == 0) return;
  if (!gemm_sl_supported(a.M, a.Kd) || a.src_ld != a.Kd)
    throw Error(-5, "sliced stage needs ranks that are multiples of 8, <= 512, and dense source rows");
  if (fp64) launch_sl<8, double2, double>(a, t, status, s);
  else launch_sl<3, float2, float>(a, t, status, s);
}

}  // namespace dfmm
