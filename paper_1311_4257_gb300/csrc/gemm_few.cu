// Translation stage y[dst] += T_op x[src] for operators that serve only a few
// (pair, right-hand side) columns each: small bodies, the coarse levels of an
// adaptive tree, the top high-frequency level.
//
// Such a stage is bound by reading its operators once (8 columns do 8 flops per
// operator byte), while the tensor-core forms compute 128 columns whatever the
// tile holds.  One block takes 64 rows of one operator and up to 16 columns: cp.async
// streams the rows through shared memory four K chunks deep, and a thread holds one row
// and half of the columns.  Columns come in tiles of 16, since a stage lasts as long
// as its fullest operator: with one block passing over its rows once per 8 columns, up to
// 28 of them, the V list of a sphere of 2 wavelengths (316 operators of 131 KB, 8 columns on
// average) took 32 us, in tiles of 16 it takes 19 and its apply 36 (47 in split form with
// 6 us for the split).  Five blocks per SM keep all 644 in flight; three chunks deep
// the longer rows of eps 1e-6 lose what the sixth block gains (285 against 277 us, sphere of 8).
// Every output is summed in the order of the CUDA-core stage kernel
// (gemm_stage_kernel): the result is its to the bit, up to the order of the additions to dst.
#include "apply.h"
#include "pdl.h"
#include "tcgen05.cuh"

namespace dfmm {

namespace {

constexpr int FW_ROWS = 64, FW_COLS = 16, FW_THREADS = 128, FW_STAGES = 4;
constexpr int FW_NV = FW_COLS / 2;            // columns per thread: the threads are 64 rows x 2 halves of the columns
constexpr int FW_K = 16;                      // K values per chunk
constexpr int FW_LD = FW_K * 8;               // 16-byte pieces of an operator row swizzled by row: eight lanes' reads hit all banks
constexpr int FW_STAGE = (FW_ROWS + FW_COLS) * FW_LD;   // operator rows, then source columns
constexpr int FW_SMEM = FW_STAGES * FW_STAGE;

__device__ __forceinline__ void cfma(float2& c, float2 a, float2 b) {
  c.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x));
  c.y = fmaf(a.x, b.y, fmaf(a.y, b.x, c.y));
}

// one chunk: this thread's row against NV columns
template <int NV>
__device__ __forceinline__ void chunk(const unsigned char* ar, int sw, const unsigned char* x, float2 (&acc)[FW_NV]) {
#pragma unroll
  for (int k = 0; k < FW_K; k += 2) {
    const float4 av = *(const float4*)(ar + ((8 * k) ^ sw));
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const float4 bv = *(const float4*)(x + j * FW_LD + 8 * k);
      cfma(acc[j], make_float2(av.x, av.y), make_float2(bv.x, bv.y));
      cfma(acc[j], make_float2(av.z, av.w), make_float2(bv.z, bv.w));
    }
  }
}

__global__ __launch_bounds__(FW_THREADS) void gemm_few_kernel(GemmArgs a) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smem[];
  const int tid = threadIdx.x;
  const int4 tile = a.tiles[blockIdx.x];
  const int row0 = blockIdx.y * FW_ROWS;
  const float2* A = a.ops + (size_t)tile.x * a.M * a.Kd;
  const int ncol = tile.z * a.nrhs, nchunk = (a.Kd + FW_K - 1) / FW_K;
  const uint32_t mg = tc::rhs_magic(a.nrhs);
  const uint32_t sbase = tc::smem_u32(smem);
  // copy roles: 8 threads per row (one 16-byte piece each), rows cr, cr + 16, ...
  const int pc = tid & 7, cr = tid >> 3;
  const uint32_t ap = (uint32_t)(pc ^ (cr & 7)) * 16;   // (cr + 16 i) & 7 = cr & 7
  const int row = tid & 63, sw = (row & 7) * 16;   // compute role: a row and half of the columns
  const float2* xp = nullptr;   // source column of this thread's piece
  if (cr < ncol) {
    const int p = tc::div_rhs(cr, mg), k = cr - p * a.nrhs;
    xp = a.src + ((int64_t)a.pairs[tile.y + p].x * a.nrhs + k) * a.src_ld;
  }
  auto fetch = [&](int ch) {
    if (ch < nchunk) {
      const uint32_t s = sbase + (uint32_t)((ch % FW_STAGES) * FW_STAGE);
      const int q = ch * FW_K + pc * 2;   // Kd is even: a piece is inside or outside
      const bool kin = q < a.Kd;
#pragma unroll
      for (int i = 0; i < FW_ROWS / 16; ++i) {
        const int r = cr + 16 * i;
        if (kin && row0 + r < a.M) tc::cp_async16(s + r * FW_LD + ap, A + (size_t)(row0 + r) * a.Kd + q);
        else tc::cp_async16_zero(s + r * FW_LD + ap, A);
      }
      if (kin && xp) tc::cp_async16(s + (FW_ROWS + cr) * FW_LD + pc * 16, xp + q);
      else tc::cp_async16_zero(s + (FW_ROWS + cr) * FW_LD + pc * 16, A);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int nh = (ncol + 1) >> 1, cg = (tid >> 6) * nh;
  const int nv = min(nh, ncol - cg);   // columns of this thread
  float2 acc[FW_NV];
#pragma unroll
  for (int j = 0; j < FW_NV; ++j) acc[j] = make_float2(0.f, 0.f);
#pragma unroll
  for (int ch = 0; ch < FW_STAGES - 1; ++ch) fetch(ch);
  for (int ch = 0; ch < nchunk; ++ch) {
    asm volatile("cp.async.wait_group %0;" ::"n"(FW_STAGES - 2) : "memory");
    __syncthreads();           // chunk ch is there, chunk ch - 1 has been consumed
    fetch(ch + FW_STAGES - 1);
    const unsigned char* s = smem + (ch % FW_STAGES) * FW_STAGE;
    const unsigned char* ar = s + row * FW_LD;
    const unsigned char* x = s + (FW_ROWS + cg) * FW_LD;
    switch (nv) {   // uniform over a warp
      case 1: chunk<1>(ar, sw, x, acc); break;
      case 2: chunk<2>(ar, sw, x, acc); break;
      case 3: chunk<3>(ar, sw, x, acc); break;
      case 4: chunk<4>(ar, sw, x, acc); break;
      case 5: chunk<5>(ar, sw, x, acc); break;
      case 6: chunk<6>(ar, sw, x, acc); break;
      case 7: chunk<7>(ar, sw, x, acc); break;
      case 8: chunk<8>(ar, sw, x, acc); break;
      default: break;
    }
  }
  if (row0 + row < a.M) {
#pragma unroll
    for (int j = 0; j < FW_NV; ++j)
      if (j < nv) {
        const int p = tc::div_rhs(cg + j, mg), k = cg + j - p * a.nrhs;
        float2* d = a.dst + ((int64_t)a.pairs[tile.y + p].y * a.nrhs + k) * a.dst_ld + row0 + row;
        tc::red_add2((float*)d, acc[j].x, acc[j].y);
      }
  }
}

}  // namespace

int gemm_few_columns() { return FW_COLS; }

void launch_gemm_stage_few(const GemmArgs& a, LaunchStream s) {
  if (a.ntiles == 0) return;
  if (a.Kd % 8 || a.src_ld % 2) throw Error(-5, "few-column stage needs source ranks that are multiples of 8");
  if (a.nrhs > FW_COLS) throw Error(-5, "few-column stage takes up to 16 right-hand sides");
  const dim3 grid((unsigned)a.ntiles, (unsigned)((a.M + FW_ROWS - 1) / FW_ROWS));
  launch_pdl(gemm_few_kernel, grid, FW_THREADS, FW_SMEM, s, a);
  DFMM_CUDA(cudaGetLastError());
}

}  // namespace dfmm
