// Split-complex tensor-core form of the translation stage y[dst] += T_op x[src]
// (M2L and the other translations of the same gather / GEMM / scatter-add
// shape), for target ranks up to 256 (FP16 split; 128 for the others).
//
// A complex product y = T x is four real products,
//     Re y = Tr xr - Ti xi,     Im y = Ti xr + Tr xi,
// each a GEMM with N = r_t (the target rank) and K = r_s.  The operator is
// stored as its real and imaginary parts once each, half the bytes of the
// real-block form [[Tr, -Ti], [Ti, Tr]] that m2l_tc.cu streams per tile, and
// the source rows are split into their real and imaginary halves.  The minus
// sign is the MMA's negate-A flag.
//
//  * One CTA computes a tile of 128 gathered columns (pairs x right-hand
//    sides) against one operator (a block of n <= 128 of its outputs beyond rank
//    128), with tcgen05.mma kind::f16, M = 128, K = 16, FP32 accumulation in
//    tensor memory.
//  * Scaled split as in m2l_tc.cu: x / s = hi + lo per source row and
//    T / t = hi + lo per operator, in one of three element types (KIND):
//    FP16 (kind::f16, the default), BF16 (kind::f16 with BF16 operands:
//    "3xBF16", about 16 bits) or TF32 (kind::tf32: "3xTF32", about 22 bits,
//    half the FP16 rate).  Every tile is 128 bytes per row and K step 32
//    bytes whatever the type, so one layout serves all three.  The products are
//    hi hi and the cross terms hi lo + lo hi.  The hi hi products go to the
//    accumulators Re Y, Im Y, and the
//    cross terms either to a second pair re y, im y, added in
//    FP32 by the epilogue (ONE = false: tensor-core accumulation truncates, so
//    the small terms keep their own accumulators; 4 n <= 512 tensor-memory
//    columns, one tile at a time), or into Re Y, Im Y as well (ONE = true, the
//    automatic choice at eps >= 1e-5: 2 n columns per buffer and two
//    buffers, so that a tile's MMAs overlap the previous tile's epilogue).
//  * A K chunk is one 128-byte line of each of xr lo, xi lo, xr hi, xi hi per
//    row and lands as one row of a 128-byte-swizzled tile.  cp.async takes a
//    shared-memory pass per line that an instruction touches and per 16-byte
//    piece that meets another in a bank: 64-byte pieces in the unswizzled
//    layout took 32 passes per 512 bytes, and now it is 4.  That pipe also
//    carries the epilogue's reductions, so both waited for it.
//  * Re and Im lie side by side in tensor memory and Tr, Ti in the operator
//    chunk, so xr is multiplied by both with one MMA of N = 2 n: 96 clocks of
//    operand reads for 128 of products, where two of N = 128 read as long as they
//    multiply and leave the copies no room.
//  * Epilogue: the .16x256b tensor-memory shape gives a thread two
//    consecutive outputs p, p + 1 of a column in each accumulator, i.e. the
//    interleaved target components 2p .. 2p + 3: one 16-byte reduction
//    (red.global.add.v4.f32), and one warp instruction covers 8 target rows x
//    64 contiguous bytes.  Eight warps: 4.35 against 4.54 ms with four on the apply below.
//
//  * The MMA warp issues converged, from an elected lane (tcgen05.cuh): from one
//    diverged thread an MMA took 115 to 140 clocks to issue, more than most take to run.
//
// Measured, sphere of 64 wavelengths, eps 1e-5 (N = 1,286,796): all
// translations 5.27 -> 3.13 ms (228 -> 378 TFLOP/s useful, of 655 at the measured
// FP16 rate and three products), the apply 6.40 -> 4.22 ms; ellipsoid of 32 with 16
// right-hand sides, whose rank 144 stages took the real-block form: 6.53 -> 3.73
// ms.  Of these the warp-wide issue gave 4.31 -> 4.22 and 4.02 -> 3.73 ms.  Role timers: a
// tile takes 11k clocks, 6.1k of them MMAs at the unhindered rate and 7.4k the
// epilogue's reductions into L2 (128 KB a tile at 5 TB/s over the chip); copies,
// operand reads and reductions share the SM's memory pipe, and that is what bounds it.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "apply.h"
#include "pdl.h"
#include "per_device.h"
#include "tcgen05.cuh"

namespace dfmm {

namespace {

using namespace tc;

constexpr int CX_M = 128;                          // gathered columns per tile
constexpr int CX_SEG = 128;                        // bytes per row of a tile: one K chunk of one half
constexpr int CX_NMAX = 128;                       // outputs per block
constexpr int CX_PRODUCERS = 128;                  // warps 0-3: gather
constexpr int CX_EPI = 8;                          // epilogue warps
constexpr int CX_MMA_WARP = 4 + CX_EPI;            // warps 4 ..: epilogue; the last: MMA issuer
constexpr int CX_THREADS = 32 * (CX_MMA_WARP + 1);
constexpr int CX_NA = 6, CX_NB = 2;                // ring slots: gathered tiles, operator chunks
constexpr int CX_TILE = CX_M * CX_SEG;             // 16 KB: one of xr hi, xr lo, xi hi, xi lo
constexpr int CX_B_MAX = 4 * CX_NMAX * CX_SEG;     // 64 KB: Tr hi, Ti hi, Tr lo, Ti lo
constexpr int CX_SMEM = CX_NA * CX_TILE + CX_NB * CX_B_MAX + 1024 + 256;
constexpr int CX_TMEM_COLS = 512;

// outputs per block for target rank M: one block up to 128, equal blocks beyond
__host__ __device__ __forceinline__ int cx_block(int M) {
  const int nb = (M + CX_NMAX - 1) / CX_NMAX;
  return ((M + nb - 1) / nb + 15) & ~15;
}

// element types: 0 = FP16, 1 = BF16, 2 = TF32 (stored as FP32 bit patterns)
template <int KIND> struct Elem;
template <> struct Elem<0> {
  using T = __half;
  static __device__ __forceinline__ void split(float v, T& h, T& l) {
    h = __float2half_rn(v);
    l = __float2half_rn(v - __half2float(h));
  }
};
template <> struct Elem<1> {
  using T = __nv_bfloat16;
  static __device__ __forceinline__ void split(float v, T& h, T& l) {
    h = __float2bfloat16_rn(v);
    l = __float2bfloat16_rn(v - __bfloat162float(h));
  }
};
__device__ __forceinline__ uint32_t to_tf32(float v) {   // round to the nearest TF32 (ties away)
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(v));
  return r;
}
template <> struct Elem<2> {
  using T = uint32_t;
  static __device__ __forceinline__ void split(float v, T& h, T& l) {
    h = to_tf32(v);
    l = to_tf32(v - __uint_as_float(h));
  }
};
template <int KIND> __host__ __device__ constexpr int elem_bytes() { return KIND == 2 ? 4 : 2; }
template <int KIND> __host__ __device__ constexpr int seg_elems() { return CX_SEG / elem_bytes<KIND>(); }   // K values per chunk
template <int KIND> __host__ __device__ constexpr int kstep_elems() { return 32 / elem_bytes<KIND>(); }    // K values per MMA

// instruction descriptor: D f32, both operands K-major, M = 128, N = n; A and
// B FP16 / BF16 (kind::f16) or TF32 (kind::tf32); neg_a negates A
template <int KIND>
__device__ __forceinline__ uint32_t idesc_cx(int n, bool neg_a) {
  const uint32_t ty = KIND == 0 ? 0u : (KIND == 1 ? 1u : 2u);
  return (1u << 4) | (ty << 7) | (ty << 10) | ((neg_a ? 1u : 0u) << 13) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(128 >> 4) << 24);
}

template <int KIND>
__device__ __forceinline__ void mma_cx(uint32_t lead, uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  if (KIND == 2)
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n @q tcgen05.mma.cta_group::1.kind::tf32 "
        "[%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(lead));
  else
    mma_f16_by(lead, d_tmem, a, b, idesc, acc);
}

// N elements (4 or 8 bytes each) of one tile row as one store
template <class T> __device__ __forceinline__ void store4(unsigned char* o, const T (&v)[4]) {
  if constexpr (sizeof(T) == 2) *(uint2*)o = *(const uint2*)v;
  else *(uint4*)o = *(const uint4*)v;
}

// Source rows (r complex values, r a multiple of 16) -> scaled hi / lo rows, one
// power-of-two scale per row: per K chunk of 128 bytes the pieces xr lo, xi lo,
// xr hi, xi hi, in the order the MMAs take them (the last chunk's pieces are as
// long as what is left; a row takes 8 r bytes, 16 r for TF32).  One warp per row, four complex
// values per lane and step.
template <int KIND>
__global__ __launch_bounds__(256) void split_cx_kernel(const float* x, int64_t rows, int r, unsigned char* out, float* scale) {
  pdl_begin();
  using E = Elem<KIND>;
  using T = typename E::T;
  constexpr int EB = elem_bytes<KIND>(), BKE = seg_elems<KIND>();
  const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  const float4* xr = (const float4*)(x + row * 2 * r);
  // the first 128 values stay in registers; longer rows are read again from L1
  float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = v0;
  if (4 * lane < r) { v0 = xr[2 * lane]; v1 = xr[2 * lane + 1]; }
  auto amax = [](float4 a, float4 b) {
    return fmaxf(fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(a.z), fabsf(a.w))),
                 fmaxf(fmaxf(fabsf(b.x), fabsf(b.y)), fmaxf(fabsf(b.z), fabsf(b.w))));
  };
  float m = amax(v0, v1);
  for (int q = 4 * lane + 128; q < r; q += 128) m = fmaxf(m, amax(xr[q / 2], xr[q / 2 + 1]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  const float s = pow2_above(m);
  const float inv = 1.f / s;
  if (lane == 0) scale[row] = s;
  unsigned char* orow = out + row * (int64_t)(4 * r * EB);
  for (int q = 4 * lane; q < r; q += 128) {
    if (q >= 128) { v0 = xr[q / 2]; v1 = xr[q / 2 + 1]; }
    T rh[4], rl[4], ih[4], il[4];
    E::split(v0.x * inv, rh[0], rl[0]);
    E::split(v0.y * inv, ih[0], il[0]);
    E::split(v0.z * inv, rh[1], rl[1]);
    E::split(v0.w * inv, ih[1], il[1]);
    E::split(v1.x * inv, rh[2], rl[2]);
    E::split(v1.y * inv, ih[2], il[2]);
    E::split(v1.z * inv, rh[3], rl[3]);
    E::split(v1.w * inv, ih[3], il[3]);
    const int c = q / BKE, w = min(BKE, r - c * BKE) * EB;   // this chunk's piece length
    unsigned char* o = orow + c * (4 * CX_SEG) + (q - c * BKE) * EB;
    store4(o, rl);
    store4(o + w, il);
    store4(o + 2 * w, rh);
    store4(o + 3 * w, ih);
  }
}

// Operator image [op][block of outputs][K chunk][Tr hi, Ti hi, Tr lo, Ti lo][row of
// the block][128 bytes], zero beyond Kd, rows swizzled as the MMA reads them: a
// chunk is one bulk copy.  One block of threads per (op, chunk).
template <int KIND>
__global__ void op_image_cx_kernel(const float2* __restrict__ ops, const float* __restrict__ scale, int M, int Kd,
                                   int nops, unsigned char* __restrict__ img) {
  using E = Elem<KIND>;
  using T = typename E::T;
  constexpr int BKE = seg_elems<KIND>(), EB = elem_bytes<KIND>();
  const int nchunk = (Kd + BKE - 1) / BKE, n = cx_block(M);
  const int64_t g = blockIdx.x;   // (op, c)
  const int c = (int)(g % nchunk);
  const int op = (int)(g / nchunk);
  if (op >= nops) return;
  unsigned char* base = img + op * ((int64_t)nchunk * 4 * M * CX_SEG);
  const float2* Top = ops + (size_t)op * M * Kd;
  const float inv = 1.f / scale[op];
  for (int e = threadIdx.x; e < M * BKE; e += blockDim.x) {
    const int p = e / BKE, kk = e % BKE;
    const int q = c * BKE + kk;
    const int blk = p / n, row = p - blk * n, nb = min(n, M - blk * n);
    float2 t = make_float2(0.f, 0.f);
    if (q < Kd) t = Top[(size_t)p * Kd + q];
    T rh, rl, ih, il;
    E::split(t.x * inv, rh, rl);
    E::split(t.y * inv, ih, il);
    unsigned char* o = base + (int64_t)blk * n * (nchunk * 4 * CX_SEG) + (int64_t)c * (4 * CX_SEG * nb) +
                       sw128_off(row, kk * EB / 16) + kk * EB % 16;
    *(T*)o = rh;
    *(T*)(o + nb * CX_SEG) = ih;
    *(T*)(o + 2 * nb * CX_SEG) = rl;
    *(T*)(o + 3 * nb * CX_SEG) = il;
  }
}

// The stage of a tile: from the launch's stage table (tile .w), or the single
// stage of GemmArgs / TcArgs.
__device__ __forceinline__ CxStage stage_of(const GemmArgs& a, const TcArgs& t, int w) {
  if (a.stages) return a.stages[w];
  CxStage s;
  s.pairs = a.pairs;
  s.src = t.src_hi;
  s.src_scale = t.src_scale;
  s.img = t.img;
  s.op_scale = t.op_scale;
  s.dst = a.dst;
  s.nrhs = a.nrhs;
  return s;
}

// Persistent, warp-specialised stage kernel; item = (tile, block of outputs), CTA
// x takes items x, x + gridDim.x, ...
//   warps 0-3  producers: 8 threads copy one row of a tile (its 128-byte chunk of
//              xr lo, xi lo, xr hi or xi hi) with 16-byte cp.async, counted on the
//              slot's full barrier, up to CX_NA tiles ahead; thread 0 also
//              bulk-copies the operator chunk, up to CX_NB chunks ahead.
//   last warp  an elected lane issues the MMAs, commits each tile and each operator
//              chunk to their slots' empty barriers and each item to acc_full; it
//              waits for acc_empty before it overwrites the accumulators.
//   warps 4 .. epilogue: warp 4 + q reads tensor-memory lanes 32 (q % 4) ..
//              32 (q % 4) + 31 (gathered columns), adds the two accumulator pairs,
//              scales, and scatter-adds 16 bytes per thread and step; then acc_empty.
// Every wait is time-limited; on a timeout the CTA reports it, stops issuing,
// lets its own copies and MMAs land, frees its tensor memory and returns.
//
// ONE = false: two accumulator pairs (hi hi terms apart from the cross terms),
// 4 n columns, one item at a time.  ONE = true: one accumulator per
// component (2 n columns) and two tensor-memory buffers, so that the MMAs
// of an item overlap the epilogue of the previous one; the cross terms of a
// chunk then come first, while the accumulators they are truncated to are small.
template <int KIND, bool ONE>
__global__ __launch_bounds__(CX_THREADS, 1) void gemm_cx_kernel(GemmArgs a, TcArgs t, int nblk, unsigned* status) {
  pdl_begin();
  constexpr int EB = elem_bytes<KIND>(), BKE = seg_elems<KIND>(), KSTEP = kstep_elems<KIND>();
  constexpr int RSTEP = CX_PRODUCERS / 8, RPT = CX_M / RSTEP;
  extern __shared__ unsigned char smem_raw[];
  __shared__ int s_start;
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t sA = smem_u32(smem), sB = sA + CX_NA * CX_TILE;
  uint64_t* fullA = (uint64_t*)(smem + CX_NA * CX_TILE + CX_NB * CX_B_MAX);
  uint64_t* emptyA = fullA + CX_NA;
  uint64_t* fullB = emptyA + CX_NA;
  uint64_t* emptyB = fullB + CX_NB;
  uint64_t* acc_full = emptyB + CX_NB;       // [2]: one per tensor-memory buffer
  uint64_t* acc_empty = acc_full + 2;        // [2]
  uint64_t* never = acc_empty + 2;   // nothing arrives here (wait_test)
  uint32_t* tmem_slot = (uint32_t*)(never + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int M = a.M, n = cx_block(M);   // target rank; outputs per block
  const int Kh = a.Kd;                  // source rank: K of each half
  const int nchunk = (Kh + BKE - 1) / BKE;
  const int nitems = (int)a.ntiles * nblk, G = (int)gridDim.x;
  const int64_t op_row = (int64_t)nchunk * 4 * CX_SEG;   // image bytes per output

  if (tid == 0) s_start = (*(volatile unsigned*)status & kStatusTimeout) ? 0 : 1;
  __syncthreads();
  if (!s_start) return;   // an earlier CTA gave up: skip the work, hold no tensor memory
  if (tid == 0) {
    for (int i = 0; i < CX_NA; ++i) {
      mbar_init(smem_u32(&fullA[i]), CX_PRODUCERS);
      mbar_init(smem_u32(&emptyA[i]), 1);
    }
    for (int i = 0; i < CX_NB; ++i) {
      mbar_init(smem_u32(&fullB[i]), 1);
      mbar_init(smem_u32(&emptyB[i]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&acc_full[b]), 1);
      mbar_init(smem_u32(&acc_empty[b]), CX_EPI);
    }
    mbar_init(smem_u32(never), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == CX_MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(CX_TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp < CX_PRODUCERS / 32) {
    // ---------------- producers ----------------
    const int pc = tid & 7, r0 = tid >> 3;   // 16-byte piece; rows r0 + 16 q
    const uint32_t dst0 = sw128_off(r0, pc);
    const int64_t src_row = (int64_t)4 * Kh * EB;   // bytes of a split source row
    // The source row of each gathered column: (pair, right-hand side) -> source
    // state row.  The tile records and pair indices of the next item are loaded
    // while this item's chunks are issued, so their latency stays off the
    // gather's critical path.
    auto load_rows = [&](const int4& tl, int* rows, const unsigned char*& src, const unsigned char*& img) {
      const CxStage sg = stage_of(a, t, tl.w);
      src = (const unsigned char*)sg.src;
      img = (const unsigned char*)sg.img + tl.x * (op_row * M);
      const int ncol = tl.z * sg.nrhs;
      const uint32_t mg = rhs_magic(sg.nrhs);
#pragma unroll
      for (int q = 0; q < RPT; ++q) {
        const int col = r0 + q * RSTEP;
        rows[q] = -1;
        if (col < ncol) {
          const int pr = div_rhs(col, mg);
          rows[q] = sg.pairs[tl.y + pr].x * sg.nrhs + (col - pr * sg.nrhs);
        }
      }
    };
    const int4 none = make_int4(0, 0, 0, 0);
    int it = (int)blockIdx.x;
    int4 tile_n = it < nitems ? a.tiles[it / nblk] : none;
    int rows_n[RPT];
    const unsigned char *src_n = nullptr, *img_n = nullptr;
    if (it < nitems) load_rows(tile_n, rows_n, src_n, img_n);
    int4 tile_nn = it + G < nitems ? a.tiles[(it + G) / nblk] : none;
    Ring ra, rb;
    int ga = 0, gb = 0;   // slots filled so far (ga up to the ring's size: no wait on the first round)
    bool ok = true;
    for (; it < nitems && ok; it += G) {
      const int blk = it % nblk, nb = min(n, M - blk * n);
      const unsigned char* src = src_n;
      const unsigned char* img = img_n + blk * n * op_row;
      const uint32_t bb = (uint32_t)(4 * CX_SEG * nb);
      const unsigned char* srow[RPT];
#pragma unroll
      for (int q = 0; q < RPT; ++q) srow[q] = rows_n[q] >= 0 ? src + rows_n[q] * src_row + 16 * pc : nullptr;
      // prefetch: rows of the next item, record of the one after
      tile_n = tile_nn;
      if (it + G < nitems) load_rows(tile_n, rows_n, src_n, img_n);
      tile_nn = it + 2 * G < nitems ? a.tiles[(it + 2 * G) / nblk] : none;
      for (int c = 0; c < nchunk && ok; ++c) {
        if (warp == 0) {   // operator chunk: Tr hi, Ti hi, Tr lo, Ti lo
          int okw = 1;
          if (lane == 0) {
            if (gb >= CX_NB) okw = mbar_wait(smem_u32(&emptyB[rb.st]), rb.ph ^ 1u, status) ? 1 : 0;
            if (okw) {
              mbar_expect_tx(smem_u32(&fullB[rb.st]), bb);
              bulk_g2s(sB + rb.st * CX_B_MAX, img + c * (int64_t)bb, bb, smem_u32(&fullB[rb.st]));
            }
          }
          ok = __shfl_sync(0xffffffffu, okw, 0) != 0;
          if (!ok) break;
          ++gb;
          rb.next(CX_NB);
        }
        const int w = min(BKE, Kh - c * BKE) * EB;   // bytes of this chunk's pieces
        const bool kin = 16 * pc < w;
        for (int h = 0; h < 4; ++h) {   // xr lo, xi lo, xr hi, xi hi
          if (ga >= CX_NA) {   // the slot's previous tile has been consumed by the MMAs
            int okw = 0;
            if (lane == 0) okw = mbar_wait(smem_u32(&emptyA[ra.st]), ra.ph ^ 1u, status) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, okw, 0) != 0;
            if (!ok) break;
          }
          const uint32_t d = sA + ra.st * CX_TILE + dst0;
          const int off = c * (4 * CX_SEG) + h * w;
          if (kin) {
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
              if (srow[q]) cp_async16(d + q * (RSTEP * CX_SEG), srow[q] + off);
              else cp_async16_zero(d + q * (RSTEP * CX_SEG), src);
            }
          }
          asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&fullA[ra.st])) : "memory");
          ga = min(ga + 1, CX_NA);
          ra.next(CX_NA);
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (tid == 0)   // the bulk copies of the last fills have landed
      for (int q = 0; q < min(gb, CX_NB); ++q) {
        const int g = gb - 1 - q;
        mbar_wait_drain(smem_u32(&fullB[g % CX_NB]), (uint32_t)((g / CX_NB) & 1));
      }
  } else if (warp == CX_MMA_WARP) {
    // ---------------- MMA issuer ----------------
    {
      const uint32_t lead = elect_one(), tm = __reduce_max_sync(0xffffffffu, tmem);   // uniform
      Ring ra, rb;
      int last = -1, i = 0;
      uint32_t last_ph = 0;
      // wait_test: a wait that can only end by giving up; the CTA then takes the timeout path
      bool ok = !(a.wait_test && blockIdx.x == 0) || warp_wait(smem_u32(never), 0u, status);
      for (int it = (int)blockIdx.x; it < nitems && ok; it += G, ++i) {
        const int nb = min(n, M - (it % nblk) * n);
        const uint32_t i1 = idesc_cx<KIND>(nb, false), i1n = idesc_cx<KIND>(nb, true), i2 = idesc_cx<KIND>(2 * nb, false);
        // buffer of this item: ONE alternates two buffers of 2 n columns
        const int b = ONE ? (i & 1) : 0;
        const int use = ONE ? (i >> 1) : i;   // earlier items on this buffer
        const uint32_t YR = tm + (uint32_t)(b * 256), YI = YR + (uint32_t)nb;
        const uint32_t yr = ONE ? YR : YR + 2u * nb, yi = ONE ? YI : YR + 3u * nb;
        if (use > 0 && !warp_wait(smem_u32(&acc_empty[b]), (uint32_t)((use - 1) & 1), status)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // next gathered tile: its address in shared memory once it is full
        auto take = [&](uint32_t& xa, uint32_t& bar) {
          if (!warp_wait(smem_u32(&fullA[ra.st]), ra.ph, status)) return false;
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // cp.async data -> async proxy
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          xa = sA + ra.st * CX_TILE;
          bar = smem_u32(&emptyA[ra.st]);
          last = ra.st;
          last_ph = ra.ph;
          ra.next(CX_NA);
          return true;
        };
        for (int c = 0; c < nchunk; ++c) {
          uint32_t xr, xi, br, bi;
          ok = warp_wait(smem_u32(&fullB[rb.st]), rb.ph, status) && take(xr, br);
          if (!ok) break;
          const int ksteps = min(BKE, Kh - c * BKE) / KSTEP;
          // operator rows: [Tr hi | Ti hi], [Tr lo | Ti lo]; y = [Re | Im] are adjacent columns, so one
          // MMA of N = 2 n multiplies xr by both; xi takes two (Re y -= Ti xi, Im y += Tr xi)
          const uint64_t rh = smem_desc_sw128(sB + rb.st * CX_B_MAX), ih = rh + (uint64_t)(nb * CX_SEG / 16),
                         rl = ih + (uint64_t)(nb * CX_SEG / 16), il = rl + (uint64_t)(nb * CX_SEG / 16);
          const uint64_t dl = smem_desc_sw128(xr);
          // cross terms: xr lo, xi lo with T hi; xr hi, xi hi with T lo
          for (int k = 0; k < ksteps; ++k)
            mma_cx<KIND>(lead, yr, dl + 2 * k, rh + 2 * k, i2, (c > 0 || k > 0) ? 1u : 0u);
          mma_commit_by(lead, br);
          ok = take(xi, bi);
          if (!ok) break;
          const uint64_t el = smem_desc_sw128(xi);
          for (int k = 0; k < ksteps; ++k) {
            mma_cx<KIND>(lead, yr, el + 2 * k, ih + 2 * k, i1n, 1u);
            mma_cx<KIND>(lead, yi, el + 2 * k, rh + 2 * k, i1, 1u);
          }
          mma_commit_by(lead, bi);
          ok = take(xr, br);
          if (!ok) break;
          const uint64_t dh = smem_desc_sw128(xr);
          for (int k = 0; k < ksteps; ++k) mma_cx<KIND>(lead, yr, dh + 2 * k, rl + 2 * k, i2, 1u);
          ok = take(xi, bi);
          if (!ok) break;
          const uint64_t eh = smem_desc_sw128(xi);
          for (int k = 0; k < ksteps; ++k) {
            mma_cx<KIND>(lead, yr, eh + 2 * k, il + 2 * k, i1n, 1u);
            mma_cx<KIND>(lead, yi, eh + 2 * k, rl + 2 * k, i1, 1u);
          }
          // the large terms
          for (int k = 0; k < ksteps; ++k)
            mma_cx<KIND>(lead, YR, dh + 2 * k, rh + 2 * k, i2, (ONE || c > 0 || k > 0) ? 1u : 0u);
          mma_commit_by(lead, br);
          for (int k = 0; k < ksteps; ++k) {
            mma_cx<KIND>(lead, YR, eh + 2 * k, ih + 2 * k, i1n, 1u);
            mma_cx<KIND>(lead, YI, eh + 2 * k, rh + 2 * k, i1, 1u);
          }
          mma_commit_by(lead, bi);
          mma_commit_by(lead, smem_u32(&emptyB[rb.st]));
          rb.next(CX_NB);
        }
        if (!ok) break;
        mma_commit_by(lead, smem_u32(&acc_full[b]));
      }
      if (last >= 0) {   // every MMA issued so far has completed once one more commit has arrived
        mma_commit_by(lead, smem_u32(never));
        mbar_wait_drain(smem_u32(never), 0u);
      }
    }
    __syncwarp();
  } else {
    // ---------------- epilogue ----------------
    const int quarter = warp & 3, par = (warp - 4) >> 2;
    int i = 0;
    for (int it = (int)blockIdx.x; it < nitems; it += G, ++i) {
      const int4 tile = a.tiles[it / nblk];
      const int blk = it % nblk, nb = min(n, M - blk * n);
      const CxStage sg = stage_of(a, t, tile.w);
      const uint32_t mg = rhs_magic(sg.nrhs);
      constexpr int NBK = 8 / CX_EPI;   // 16-lane blocks per warp
      float* out[2 * NBK];
      float cs[2 * NBK];
#pragma unroll
      for (int h = 0; h < 2 * NBK; ++h) {   // columns 32q + 16 (par + h/2) + lane/4 + 8 (h%2)
        const int col = 32 * quarter + 16 * (par + (h >> 1)) + (lane >> 2) + 8 * (h & 1);
        out[h] = nullptr;
        cs[h] = 0.f;
        if (col < tile.z * sg.nrhs) {
          const int q = div_rhs(col, mg);
          const int2 pr = sg.pairs[tile.y + q];
          const int k = col - q * sg.nrhs;
          cs[h] = sg.src_scale[(int64_t)pr.x * sg.nrhs + k] * sg.op_scale[tile.x];
          out[h] = (float*)(sg.dst + ((int64_t)pr.y * sg.nrhs + k) * a.dst_ld) + 2 * blk * n + 4 * (lane & 3);
        }
      }
      const int b = ONE ? (i & 1) : 0;
      const int use = ONE ? (i >> 1) : i;
      int okw = 0;
      if (lane == 0) okw = mbar_wait(smem_u32(&acc_full[b]), (uint32_t)(use & 1), status) ? 1 : 0;
      okw = __shfl_sync(0xffffffffu, okw, 0);
      if (!okw) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int bk = 0; bk < NBK; ++bk) {
        const uint32_t tb = tmem + (uint32_t)(b * 256) + ((uint32_t)(32 * quarter + 16 * (par + bk)) << 16);
        float* oA = out[2 * bk];
        float* oB = out[2 * bk + 1];
        const float cA = cs[2 * bk], cB = cs[2 * bk + 1];
        for (int j0 = 0; j0 < nb; j0 += 32) {
          uint32_t vr[16], vi[16], wr[16], wi[16];
          __syncwarp();
          tmem_ld16x256_x4(tb + (uint32_t)j0, vr);
          tmem_ld16x256_x4(tb + (uint32_t)(nb + j0), vi);
          if (!ONE) {
            tmem_ld16x256_x4(tb + (uint32_t)(2 * nb + j0), wr);
            tmem_ld16x256_x4(tb + (uint32_t)(3 * nb + j0), wi);
          } else {
#pragma unroll
            for (int q = 0; q < 16; ++q) wr[q] = wi[q] = 0u;
          }
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            // this thread's outputs p = j0 + 8 j + 2 (lane % 4) + {0, 1}: target floats 2p .. 2p + 3
            if (j0 + 8 * j < nb) {
              const int f = 2 * j0 + 16 * j;
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                float* o = h ? oB : oA;
                const float cc = h ? cB : cA;
                const int r = 4 * j + 2 * h;
                const float re0 = (__uint_as_float(vr[r]) + __uint_as_float(wr[r])) * cc;
                const float im0 = (__uint_as_float(vi[r]) + __uint_as_float(wi[r])) * cc;
                const float re1 = (__uint_as_float(vr[r + 1]) + __uint_as_float(wr[r + 1])) * cc;
                const float im1 = (__uint_as_float(vi[r + 1]) + __uint_as_float(wi[r + 1])) * cc;
                if (o) red_add4(o + f, re0, im0, re1, im1);
              }
            }
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acc_empty[b])) : "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == CX_MMA_WARP)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(CX_TMEM_COLS));
}

}  // namespace

int gemm_cx_columns() { return CX_M; }

bool gemm_cx_supported(int M, int Kd, int kind) {
  return M % 16 == 0 && Kd % 16 == 0 && M >= 16 && M <= (kind == 0 ? 2 * CX_NMAX : CX_NMAX);
}

int cx_elem_bytes(int kind) { return kind == 2 ? 4 : 2; }

int64_t cx_image_bytes(int M, int Kd, int nops, int kind) {
  const int bke = CX_SEG / cx_elem_bytes(kind);
  const int nchunk = (Kd + bke - 1) / bke;
  return (int64_t)nops * nchunk * 4 * M * CX_SEG;
}

void build_cx_image(const float2* ops, int M, int Kd, int nops, void* img, float* scale, int kind, cudaStream_t s) {
  if (nops == 0) return;
  if (!gemm_cx_supported(M, Kd, kind)) throw Error(-5, "split-complex stage needs ranks that are multiples of 16, <= 256");
  compute_op_scales(ops, (int64_t)M * Kd, nops, scale, s);
  const int bke = CX_SEG / cx_elem_bytes(kind);
  const unsigned blocks = (unsigned)((int64_t)nops * ((Kd + bke - 1) / bke));
  unsigned char* p = (unsigned char*)img;
  if (kind == 0) op_image_cx_kernel<0><<<blocks, 256, 0, s>>>(ops, scale, M, Kd, nops, p);
  else if (kind == 1) op_image_cx_kernel<1><<<blocks, 256, 0, s>>>(ops, scale, M, Kd, nops, p);
  else op_image_cx_kernel<2><<<blocks, 256, 0, s>>>(ops, scale, M, Kd, nops, p);
  DFMM_CUDA(cudaGetLastError());
}

void launch_split_cx(const float2* x, int64_t rows, int r, void* out, float* scale, int kind, LaunchStream s) {
  if (rows == 0) return;
  if (r % 16) throw Error(-5, "split-complex source rows need a rank that is a multiple of 16");
  const unsigned grid = (unsigned)((rows * 32 + 255) / 256);
  const float* xf = (const float*)x;
  unsigned char* o = (unsigned char*)out;
  if (kind == 0) launch_pdl(split_cx_kernel<0>, grid, 256, 0, s, xf, rows, r, o, scale);
  else if (kind == 1) launch_pdl(split_cx_kernel<1>, grid, 256, 0, s, xf, rows, r, o, scale);
  else launch_pdl(split_cx_kernel<2>, grid, 256, 0, s, xf, rows, r, o, scale);
  DFMM_CUDA(cudaGetLastError());
}

template <int KIND, bool ONE>
void launch_cx(const GemmArgs& a, const TcArgs& t, unsigned* status, LaunchStream s) {
  static PerDevice<int> sms;   // set up with the kernel's launch attribute
  int dev = 0;
  DFMM_CUDA(cudaGetDevice(&dev));
  const int nsm = sms.get(dev, [&] {
    int n = 0;
    DFMM_CUDA(cudaFuncSetAttribute(gemm_cx_kernel<KIND, ONE>, cudaFuncAttributeMaxDynamicSharedMemorySize, CX_SMEM));
    DFMM_CUDA(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
    return n;
  });
  const int n = cx_block(a.M), nblk = (a.M + n - 1) / n;
  const int64_t items = a.ntiles * nblk;
  if (items > INT32_MAX / 2) throw Error(-5, "translation stage has too many work items");
  launch_pdl(gemm_cx_kernel<KIND, ONE>, (unsigned)std::min<int64_t>(items, nsm), CX_THREADS, CX_SMEM, s, a, t, nblk, status);
}

void launch_gemm_stage_cx(const GemmArgs& a, const TcArgs& t, unsigned* status, bool one_acc, int kind,
                          LaunchStream s) {
  if (a.ntiles == 0) return;
  if (!gemm_cx_supported(a.M, a.Kd, kind) || a.src_ld != a.Kd)
    throw Error(-5, "split-complex stage needs ranks that are multiples of 16, <= 256, and dense source rows");
  if (kind == 0) {
    if (one_acc) launch_cx<0, true>(a, t, status, s);
    else launch_cx<0, false>(a, t, status, s);
  } else if (kind == 1) {
    if (one_acc) launch_cx<1, true>(a, t, status, s);
    else launch_cx<1, false>(a, t, status, s);
  } else {
    if (one_acc) launch_cx<2, true>(a, t, status, s);
    else launch_cx<2, false>(a, t, status, s);
  }
  DFMM_CUDA(cudaGetLastError());
}

}  // namespace dfmm
