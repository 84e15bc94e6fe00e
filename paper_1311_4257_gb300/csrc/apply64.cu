// FP64 forms of the apply-time kernels, for tolerances below what FP32
// arithmetic reaches (eps < 1e-6, down to the 1e-8 level of Table 1).
//
// The argument structs are those of the FP32 kernels (apply.h); in this form
// every complex array they name (operators, rows, states, densities,
// potentials) holds complex128 (double2) elements at the same indices.  Points
// are rebuilt in FP64 from their double-float local coordinates (hi + lo
// carries 48 significant bits, exact in a double) and centre offsets are exact
// dyadic values.  The translations of this form run in slices on the tensor
// cores (m2l_sl.cu); the kernels here are bound by the FP64 pipe, which takes 16
// clocks per warp instruction, so they count FP64 instructions.  Sphere of 8
// wavelengths, eps 1e-8 (N = 20,106): near field 1.75 -> 0.50 ms (35 FP64
// instructions per interaction: 0.32 ms), P2M 0.217 -> 0.061, L2P 0.097 -> 0.054;
// cube of 4, 4 right-hand sides: P2L 1.39 -> 0.69, P2M 1.26 -> 0.16 ms.
#include <algorithm>
#include <type_traits>

#include "apply.h"
#include "pdl.h"

namespace dfmm {

namespace {

__device__ __forceinline__ const double2* c128(const float2* p) { return reinterpret_cast<const double2*>(p); }
__device__ __forceinline__ double2* c128(float2* p) { return reinterpret_cast<double2*>(p); }

__device__ __forceinline__ void cfma(double2& acc, double2 a, double2 b) {
  acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
  acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
}

constexpr int kTrig = 256;   // table of exp(2 pi i k / 256)

__global__ void trig_table_kernel(double2* t) {
  double sn, cs;
  sincospi(threadIdx.x * (2.0 / kTrig), &sn, &cs);
  t[threadIdx.x] = make_double2(cs, sn);
}

// exp(2 pi i d) / d for the difference (dx, dy, dz); coincident points give 0.
// 28 FP64 instructions, where sqrt, a division and sincospi took about 190:
//  * 1 / d from the special-function unit's rsqrt (20 bits) by one third-order
//    step, y (1 + e / 2 + 3 e^2 / 8) with e = 1 - r2 y^2 (the next term is below
//    2^-60), and d = r2 / d by one Newton step, both to about an ulp;
//  * d = k / 256 + r with |2 pi r| <= 0.0123: exp(2 pi i k / 256) from the table,
//    sine and cosine of 2 pi r by their Taylor series to r^5 and r^6 (the next
//    terms are below 1e-17).
// Distances are below 2^13 (K <= 4096); those below 2^-500 take the library functions.
__device__ __forceinline__ double2 green64(double dx, double dy, double dz, const double2* trig) {
  const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
  const uint32_t ex = (uint32_t)__double2hiint(r2) >> 20;
  if (ex - 23u > 2000u) {   // also zero, infinity and NaN
    if (!(r2 > 0.0)) return make_double2(0.0, 0.0);
    const double d = sqrt(r2), inv = 1.0 / d;
    double sn, cs;
    sincospi(2.0 * d, &sn, &cs);
    return make_double2(cs * inv, sn * inv);
  }
  double y0;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(r2));
  const double e = fma(-(r2 * y0), y0, 1.0);
  const double inv = fma(y0 * e, fma(e, 0.375, 0.5), y0);
  const double d0 = r2 * inv;
  const double d = fma(0.5 * inv, fma(-d0, d0, r2), d0);
  constexpr double kRound = 6755399441055744.0;   // 1.5 * 2^52: adding it rounds to an integer
  constexpr double p2 = 6.283185307179586476925;
  constexpr double s3 = -p2 * p2 * p2 / 6, s5 = p2 * p2 * p2 * p2 * p2 / 120;
  constexpr double c2 = -p2 * p2 / 2, c4 = p2 * p2 * p2 * p2 / 24, c6 = -p2 * p2 * p2 * p2 * p2 * p2 / 720;
  const double t = fma(d, (double)kTrig, kRound);
  const double2 w = trig[__double2loint(t) & (kTrig - 1)];
  const double r = fma(t - kRound, -1.0 / kTrig, d);
  const double q = r * r;
  const double sr = r * fma(q, fma(q, s5, s3), p2);
  const double cr = q * fma(q, fma(q, c6, c4), c2);   // cos - 1
  const double cs = fma(w.x, cr, fma(-w.y, sr, w.x));
  const double sn = fma(w.y, cr, fma(w.x, sr, w.y));
  return make_double2(cs * inv, sn * inv);
}

// FP64 local coordinates of sorted point j, shifted by sh
__device__ __forceinline__ double3 point64(const float4* hi, const float4* lo, int64_t j, float4 sh) {
  const float4 h = hi[j], l = lo[j];
  return make_double3(((double)h.x + (double)l.x) + (double)sh.x, ((double)h.y + (double)l.y) + (double)sh.y,
                      ((double)h.z + (double)l.z) + (double)sh.z);
}

__device__ __forceinline__ void add_to(double2* p, double2 v) {
  atomicAdd(&p->x, v.x);
  atomicAdd(&p->y, v.y);
}

// y[dst] += T_op x[src] over a stage's pairs: one CTA computes a 64-row x
// 64-column block of T_op X (columns = gathered source rows x right-hand
// sides) and adds it into the target rows with FP64 atomics.  Where a product's columns are divided over
// several operators (P2L), gridDim.z of them with part_pairs pairs each, the tiles are the first one's.
constexpr int GM = 64, GN = 64, GK = 8;

__global__ __launch_bounds__(256) void gemm64_kernel(GemmArgs a, int64_t part_pairs) {
  pdl_begin();
  __shared__ double2 As[GK][GM + 1];
  __shared__ double2 Bs[GK][GN + 1];
  __shared__ const double2* srcp[GN];
  __shared__ double2* dstp[GN];
  const int tid = threadIdx.x;
  const int4 tile = a.tiles[blockIdx.x];
  const double2* A = c128(a.ops) + (size_t)(tile.x + blockIdx.z) * a.M * a.Kd;
  const int2* pairs = a.pairs + blockIdx.z * part_pairs;
  const int row0 = blockIdx.y * GM;
  const int ncol = tile.z * a.nrhs;
  if (tid < GN) {
    const double2* sp = nullptr;
    double2* dp = nullptr;
    if (tid < ncol) {
      const int p = tile.y + tid / a.nrhs, k = tid % a.nrhs;
      const int2 pr = pairs[p];
      sp = c128(a.src) + ((int64_t)pr.x * a.nrhs + k) * a.src_ld;
      dp = c128(a.dst) + ((int64_t)pr.y * a.nrhs + k) * a.dst_ld;
    }
    srcp[tid] = sp;
    dstp[tid] = dp;
  }
  __syncthreads();
  const int ty = tid / 16, tx = tid % 16;
  double2 acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_double2(0.0, 0.0);
  for (int k0 = 0; k0 < a.Kd; k0 += GK) {
    for (int e = tid; e < GM * GK; e += 256) {
      const int i = e / GK, kk = e % GK;
      const int r = row0 + i, kc = k0 + kk;
      As[kk][i] = (r < a.M && kc < a.Kd) ? A[(size_t)r * a.Kd + kc] : make_double2(0.0, 0.0);
    }
    for (int e = tid; e < GN * GK; e += 256) {
      const int c = e / GK, kk = e % GK;
      const int kc = k0 + kk;
      Bs[kk][c] = (c < ncol && kc < a.Kd) ? srcp[c][kc] : make_double2(0.0, 0.0);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) {
      double2 av[4], bv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) av[i] = As[kk][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) bv[j] = Bs[kk][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) cfma(acc[i][j], av[i], bv[j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = tx * 4 + j;
    if (c >= ncol) continue;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = row0 + ty * 4 + i;
      if (r < a.M) add_to(dstp[c] + r, acc[i][j]);
    }
  }
}

__global__ void permute_out64_kernel(const double2* us, const int32_t* perm, int64_t N, int nrhs, double2* u) {
  pdl_begin();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= N * nrhs) return;
  u[(e % nrhs) * N + perm[e / nrhs]] = us[e];
}

constexpr int C64_T = 128;   // threads of the check-point and near-field kernels
// NR: right-hand sides per pass, a template parameter (1, 2 or 4): instructions that are
// predicated off for a missing right-hand side take the FP64 pipe all the same
template <class F>
void by_rhs(int nrhs, F&& f) {
  if (nrhs == 1) f(std::integral_constant<int, 1>());
  else if (nrhs == 2) f(std::integral_constant<int, 2>());
  else f(std::integral_constant<int, 4>());
}

// Check-point potentials of a job's source points (the P2L sample of Eq. 6): one
// block per (job, C64_T check points), one thread per check point, sources staged in
// shared memory C64_T at a time; padding entries up to ld are written as zeros.
template <int NR>
__global__ __launch_bounds__(C64_T) void p2c64_kernel(P2CArgs a) {
  pdl_begin();
  __shared__ double3 sp[C64_T];
  __shared__ double2 sf[C64_T][NR];
  __shared__ double2 trig[kTrig];
  for (int k = threadIdx.x; k < kTrig; k += C64_T) trig[k] = a.trig[k];   // read after the first barrier below
  const int4 job = a.jobs[blockIdx.x];
  const float4 sh = a.shifts[job.w];
  const double2* fs = c128(a.fs);
  const int half = a.ld / a.halves;   // the row's length where its halves are rows of their own
  double2* out = c128(a.out) + (int64_t)job.z * a.nrhs * a.ld;
  const int p = blockIdx.y * C64_T + threadIdx.x;
  const bool live = p < a.nchk;
  const double cx = live ? a.chk64[3 * p] : 0.0, cy = live ? a.chk64[3 * p + 1] : 0.0,
               cz = live ? a.chk64[3 * p + 2] : 0.0;
  for (int r0 = 0; r0 < a.nrhs; r0 += NR) {
    const int nr = min(NR, a.nrhs - r0);
    double2 acc[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) acc[k] = make_double2(0.0, 0.0);
    for (int i0 = 0; i0 < job.y; i0 += C64_T) {
      const int ni = min(C64_T, job.y - i0);
      __syncthreads();
      if (threadIdx.x < ni) {
        const int64_t j = (int64_t)job.x + i0 + threadIdx.x;
        sp[threadIdx.x] = point64(a.pts, a.pts_lo, j, sh);
#pragma unroll
        for (int k = 0; k < NR; ++k) sf[threadIdx.x][k] = k < nr ? fs[j * a.nrhs + r0 + k] : make_double2(0.0, 0.0);
      }
      __syncthreads();
      if (live)
        for (int i = 0; i < ni; ++i) {
          const double3 v = sp[i];
          const double2 g = green64(cx - v.x, cy - v.y, cz - v.z, trig);
#pragma unroll
          for (int k = 0; k < NR; ++k) cfma(acc[k], g, sf[i][k]);
        }
    }
    if (p < a.ld)
      for (int k = 0; k < nr; ++k)
        out[(int64_t)((p / half) * a.nrhs + r0 + k) * half + p % half] = live ? acc[k] : make_double2(0.0, 0.0);
  }
}

// Dot products of point rows with states: row r (one warp) gives
// us[point][k] += sum_q rows[r][q] state[srow][k][q].  rows_kernel form (jobs
// of consecutive rows) for M2P, map form (one (point, state row) per row) for L2P.

// Sums of N = 2 NR values over the warp: every exchange halves the values a lane holds, so
// N values take N - 1 + (5 - log2 N) additions per lane (N: 5 N).  Returns the sum
// of value warp_slot<N>() on every lane.
template <int N> __device__ __forceinline__ int warp_slot() {
  const int lane = threadIdx.x & 31;
  return lane / (32 / N);
}
template <int N>
__device__ __forceinline__ double warp_sums(double (&v)[N]) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int n = N / 2; n > 0; n >>= 1, o >>= 1)
#pragma unroll
    for (int j = 0; j < n; ++j) {
      const bool up = lane & o;
      const double mine = up ? v[j + n] : v[j], theirs = up ? v[j] : v[j + n];
      v[j] = mine + __shfl_xor_sync(0xffffffffu, theirs, o);
    }
  for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  return v[0];
}

constexpr int R64_MAX = 512;         // largest rank of the FP64 row kernels

template <int NR>
__device__ __forceinline__ void row_dot(const double2* row, const double2* st, int R, int nrhs, double2* u) {
  const int lane = threadIdx.x & 31;
  for (int k0 = 0; k0 < nrhs; k0 += NR) {
    double2 sum[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) sum[k] = make_double2(0.0, 0.0);
#pragma unroll 4
    for (int q = lane; q < R; q += 32) {
      const double2 rv = row[q];
#pragma unroll
      for (int k = 0; k < NR; ++k)   // a missing right-hand side repeats the last one
        cfma(sum[k], rv, st[(int64_t)min(k0 + k, nrhs - 1) * R + q]);
    }
    __syncwarp();
    double v[2 * NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) { v[2 * k] = sum[k].x; v[2 * k + 1] = sum[k].y; }
    const double t = warp_sums<2 * NR>(v);
    const int slot = warp_slot<2 * NR>();
    if (lane % (16 / NR) == 0 && k0 + (slot >> 1) < nrhs) atomicAdd((double*)(u + k0) + slot, t);
  }
}

template <int NR>
__global__ __launch_bounds__(256) void rows64_kernel(RowsArgs a) {
  pdl_begin();
  const int4 job = a.jobs[blockIdx.x];
  const int warp = threadIdx.x / 32;
  const double2* st = c128(a.state) + (int64_t)job.w * a.nrhs * a.R;
  for (int i = warp; i < job.y; i += 8)
    row_dot<NR>(c128(a.rows) + (int64_t)(job.z + i) * a.R, st, a.R, a.nrhs, c128(a.us) + (int64_t)(job.x + i) * a.nrhs);
}

template <int NR>
__global__ __launch_bounds__(256) void l2p64_kernel(const __grid_constant__ L2PArgs a) {
  pdl_begin();
  const L2PLevel& g = a.lv[level_of(a, blockIdx.x)];
  const int64_t r = ((int64_t)(blockIdx.x - g.block0) * blockDim.x + threadIdx.x) >> 5;
  if (r >= g.nrows) return;
  const int2 m = g.map[r];
  const int R = g.R;
  row_dot<NR>(c128(g.rows) + r * R, c128(g.state) + (int64_t)m.y * a.nrhs * R, R, a.nrhs,
              c128(a.us) + (int64_t)m.x * a.nrhs);
}

// P2M through rows: state[box][k][q] = sum_i rows[row + i][q] fs[first + i][k].  One
// block per (leaf, 128 state entries), a thread per entry; NR right-hand
// sides per pass over the rows, four rows loaded ahead (one warp per leaf left
// small bodies two warps per SM).
template <int NR>
__global__ __launch_bounds__(C64_T) void p2m64_kernel(const __grid_constant__ P2MRowsArgs a) {
  pdl_begin();
  const P2MLevel& g = a.lv[level_of(a, blockIdx.x)];
  const int R = g.R, q = blockIdx.y * C64_T + threadIdx.x;
  if (q >= R) return;
  const int4 job = g.jobs[blockIdx.x - g.block0];
  const double2* row = c128(g.rows) + (int64_t)job.z * R + q;
  double2* st = c128(g.state) + (int64_t)job.w * a.nrhs * R + q;
  for (int k0 = 0; k0 < a.nrhs; k0 += NR) {
    const double2* f = c128(a.fs) + (int64_t)job.x * a.nrhs;
    double2 acc[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) acc[k] = make_double2(0.0, 0.0);
    int i = 0;
    for (; i + 4 <= job.y; i += 4) {
      double2 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = __ldcs(row + (int64_t)(i + j) * R);
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int k = 0; k < NR; ++k) cfma(acc[k], v[j], f[(int64_t)(i + j) * a.nrhs + min(k0 + k, a.nrhs - 1)]);
    }
    for (; i < job.y; ++i) {
      const double2 v = __ldcs(row + (int64_t)i * R);
#pragma unroll
      for (int k = 0; k < NR; ++k) cfma(acc[k], v, f[(int64_t)i * a.nrhs + min(k0 + k, a.nrhs - 1)]);
    }
#pragma unroll
    for (int k = 0; k < NR; ++k)
      if (k0 + k < a.nrhs) st[(int64_t)(k0 + k) * R] = acc[k];
  }
}

// Near field (U lists, Eq. 1 directly): gridDim.y blocks per target leaf, which take its
// list's entries in turn (leaves differ by a factor of ten in work).  The threads form groups
// of one thread per target (up to C64_T at a time); the staged sources, shifted into
// the target leaf's frame, are dealt to the groups in turn and the groups' sums
// added at the end, so that a leaf of a dozen points fills the block.
template <int NR>
__global__ __launch_bounds__(C64_T) void p2p64_kernel(P2PArgs a) {
  pdl_begin();
  __shared__ double3 sp[C64_T];
  __shared__ double2 sf[C64_T][NR];
  __shared__ double2 red[C64_T][NR];
  __shared__ double2 trig[kTrig];
  const int2 lr = a.leaf_range[blockIdx.x];
  const int64_t u0 = a.u_off[blockIdx.x], u1 = a.u_off[blockIdx.x + 1];
  const double2* fs = c128(a.fs);
  double2* us = c128(a.us);
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int k = threadIdx.x; k < kTrig; k += C64_T) trig[k] = a.trig[k];   // read after the first barrier below
  for (int t0 = 0; t0 < lr.y; t0 += C64_T) {
    const int nt = min(C64_T, lr.y - t0), ngrp = C64_T / nt;
    const int grp = threadIdx.x / nt, ti = threadIdx.x - grp * nt;
    const bool live = grp < ngrp;
    const double3 x = point64(a.pts, a.pts_lo, lr.x + t0 + ti, zero);
    for (int r0 = 0; r0 < a.nrhs; r0 += NR) {
      const int nr = min(NR, a.nrhs - r0);
      double2 acc[NR];
#pragma unroll
      for (int k = 0; k < NR; ++k) acc[k] = make_double2(0.0, 0.0);
      // the lists' points in order, C64_T at a time: entry e, offset i within it
      int64_t e = u0 + blockIdx.y;
      int i = 0;
      while (e < u1) {
        __syncthreads();   // the previous chunk (and the previous pass's sums) are consumed
        int fill = 0;
        while (e < u1 && fill < C64_T) {   // uniform over the block
          const int4 ue = a.u_src[e];
          const int n = min(ue.y - i, C64_T - fill);
          const int q = (int)threadIdx.x - fill;
          if (q >= 0 && q < n) {
            const int64_t j = (int64_t)ue.x + i + q;
            sp[threadIdx.x] = point64(a.pts, a.pts_lo, j, a.u_shift[e]);
#pragma unroll
            for (int k = 0; k < NR; ++k)
              sf[threadIdx.x][k] = k < nr ? fs[j * a.nrhs + r0 + k] : make_double2(0.0, 0.0);
          }
          fill += n;
          i += n;
          if (i == ue.y) { e += gridDim.y; i = 0; }
        }
        __syncthreads();
        if (live)
          for (int q = grp; q < fill; q += ngrp) {
            const double3 v = sp[q];
            const double2 g = green64(x.x - v.x, x.y - v.y, x.z - v.z, trig);
#pragma unroll
            for (int k = 0; k < NR; ++k)
              cfma(acc[k], g, sf[q][k]);
          }
      }
#pragma unroll
      for (int k = 0; k < NR; ++k) red[threadIdx.x][k] = acc[k];
      __syncthreads();
      if (threadIdx.x < nt)
        for (int k = 0; k < nr; ++k) {
          double2 sum = red[threadIdx.x][k];
          for (int g = 1; g < ngrp; ++g) {
            const double2 v = red[g * nt + threadIdx.x][k];
            sum.x += v.x;
            sum.y += v.y;
          }
          add_to(us + (int64_t)(lr.x + t0 + threadIdx.x) * a.nrhs + r0 + k, sum);
        }
    }
  }
}

void check_rank(int R) {
  if (R > R64_MAX || R < 1) throw Error(-5, "representation rank of the FP64 form must be in [1, 512]");
}

}  // namespace

void launch_gemm_stage64(const GemmArgs& a, int parts, int64_t part_pairs, LaunchStream s) {
  if (a.ntiles == 0) return;
  const dim3 grid((unsigned)a.ntiles, (unsigned)((a.M + GM - 1) / GM), (unsigned)parts);
  launch_pdl(gemm64_kernel, grid, 256, 0, s, a, part_pairs);
  DFMM_CUDA(cudaGetLastError());
}

int trig_table_bytes() { return kTrig * (int)sizeof(double2); }

void build_trig_table(void* t, cudaStream_t s) {
  trig_table_kernel<<<1, kTrig, 0, s>>>((double2*)t);
  DFMM_CUDA(cudaGetLastError());
}

void launch_permute_out64(const float2* us, const int32_t* perm, int64_t N, int nrhs, float2* u, LaunchStream s) {
  const int64_t n = N * nrhs;
  launch_pdl(permute_out64_kernel, (unsigned)((n + 255) / 256), 256, 0, s, (const double2*)us, perm, N, nrhs, (double2*)u);
  DFMM_CUDA(cudaGetLastError());
}

void launch_p2c64(const P2CArgs& a, LaunchStream s) {
  if (a.njobs == 0) return;
  if (!a.chk64 || !a.pts_lo || !a.trig) throw Error(-5, "FP64 check-point evaluation needs FP64 check points");
  const dim3 grid((unsigned)a.njobs, (unsigned)((a.ld + C64_T - 1) / C64_T));
  by_rhs(a.nrhs, [&](auto nr) { launch_pdl(p2c64_kernel<nr()>, grid, C64_T, 0, s, a); });
  DFMM_CUDA(cudaGetLastError());
}

void launch_rows64(const RowsArgs& a, LaunchStream s) {
  if (a.njobs == 0) return;
  check_rank(a.R);
  by_rhs(a.nrhs, [&](auto nr) { launch_pdl(rows64_kernel<nr()>, (unsigned)a.njobs, 256, 0, s, a); });
  DFMM_CUDA(cudaGetLastError());
}

void launch_l2p64(const L2PArgs& a, LaunchStream s) {
  for (int l = 0; l < a.nlv; ++l) check_rank(a.lv[l].R);
  L2PArgs p;
  const unsigned grid = place_levels(a, p, [](const L2PLevel&) { return true; },
                                     [](const L2PLevel& g) { return (g.nrows + 7) / 8; });
  if (grid == 0) return;
  by_rhs(a.nrhs, [&](auto nr) { launch_pdl(l2p64_kernel<nr()>, grid, 256, 0, s, p); });
  DFMM_CUDA(cudaGetLastError());
}

void launch_p2m_rows64(const P2MRowsArgs& a, LaunchStream s) {
  int R = 0;
  for (int l = 0; l < a.nlv; ++l) {
    check_rank(a.lv[l].R);
    R = std::max(R, a.lv[l].R);
  }
  P2MRowsArgs p;
  const unsigned n = place_levels(a, p, [](const P2MLevel&) { return true; },
                                  [](const P2MLevel& g) { return g.njobs; });
  if (n == 0) return;
  const dim3 grid(n, (unsigned)((R + C64_T - 1) / C64_T));
  by_rhs(a.nrhs, [&](auto nr) { launch_pdl(p2m64_kernel<nr()>, grid, C64_T, 0, s, p); });
  DFMM_CUDA(cudaGetLastError());
}

void launch_p2p64(const P2PArgs& a, LaunchStream s) {
  if (a.nleaves == 0) return;
  // enough blocks for the SMs to even out: four per leaf where the leaves alone are few
  const dim3 grid((unsigned)a.nleaves, a.nleaves < 152 * 32 ? 4u : 1u);
  by_rhs(a.nrhs, [&](auto nr) { launch_pdl(p2p64_kernel<nr()>, grid, C64_T, 0, s, a); });
  DFMM_CUDA(cudaGetLastError());
}

}  // namespace dfmm
