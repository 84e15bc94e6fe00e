// Translation stage y[dst] += T_op x[src] for operators that serve only a few
// (pair, right-hand side) columns each: small bodies, the coarse levels of an
// adaptive tree, the top high-frequency level.
//
// Such a stage is bound by reading its operators once (8 columns do 8 flops per
// operator byte), while the tensor-core forms compute 128 columns whatever the
// tile holds.  One block takes 64 rows of one operator: cp.async streams the
// rows through shared memory four K chunks deep, a thread holds one row and up
// to 4 columns, and columns beyond 8 take another pass.  Every output is summed
// in the order of the CUDA-core stage kernel (gemm_stage_kernel): the result is
// its to the bit, up to the order of the additions to dst.
#include "apply.h"
#include "pdl.h"
#include "tcgen05.cuh"

namespace dfmm {

namespace {

constexpr int FW_ROWS = 64, FW_COLS = 8, FW_THREADS = 128, FW_STAGES = 4;
constexpr int FW_K = 16;                      // K values per chunk
constexpr int FW_LD = FW_K * 8 + 16;          // padded: eight lanes' 16-byte reads of a chunk column hit all banks
constexpr int FW_STAGE = (FW_ROWS + FW_COLS) * FW_LD;   // operator rows, then source columns
constexpr int FW_SMEM = FW_STAGES * FW_STAGE;

__device__ __forceinline__ void cfma(float2& c, float2 a, float2 b) {
  c.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x));
  c.y = fmaf(a.x, b.y, fmaf(a.y, b.x, c.y));
}

// one chunk: this thread's row against NV columns
template <int NV>
__device__ __forceinline__ void chunk(const unsigned char* ar, const unsigned char* x, float2 (&acc)[4]) {
#pragma unroll
  for (int k = 0; k < FW_K; k += 2) {
    const float4 av = *(const float4*)(ar + 8 * k);
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
  // compute roles: row and four columns
  const int row = tid & 63, cg = (tid >> 6) * 4;
  for (int c0 = 0; c0 < ncol; c0 += FW_COLS) {
    const float2* xp = nullptr;   // source column of this thread's piece
    if (cr < FW_COLS && c0 + cr < ncol) {
      const int p = tc::div_rhs(c0 + cr, mg), k = c0 + cr - p * a.nrhs;
      xp = a.src + ((int64_t)a.pairs[tile.y + p].x * a.nrhs + k) * a.src_ld;
    }
    auto fetch = [&](int ch) {
      if (ch < nchunk) {
        const uint32_t s = sbase + (uint32_t)((ch % FW_STAGES) * FW_STAGE + pc * 16);
        const int q = ch * FW_K + pc * 2;   // Kd is even: a piece is inside or outside
        const bool kin = q < a.Kd;
#pragma unroll
        for (int i = 0; i < FW_ROWS / 16; ++i) {
          const int r = cr + 16 * i;
          if (kin && row0 + r < a.M) tc::cp_async16(s + r * FW_LD, A + (size_t)(row0 + r) * a.Kd + q);
          else tc::cp_async16_zero(s + r * FW_LD, A);
        }
        if (cr < FW_COLS) {
          if (kin && xp) tc::cp_async16(s + (FW_ROWS + cr) * FW_LD, xp + q);
          else tc::cp_async16_zero(s + (FW_ROWS + cr) * FW_LD, A);
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int nv = min(4, ncol - c0 - cg);   // columns of this thread (none if <= 0)
    float2 acc[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[j] = make_float2(0.f, 0.f);
#pragma unroll
    for (int ch = 0; ch < FW_STAGES - 1; ++ch) fetch(ch);
    for (int ch = 0; ch < nchunk; ++ch) {
      asm volatile("cp.async.wait_group %0;" ::"n"(FW_STAGES - 2) : "memory");
      __syncthreads();           // chunk ch is there, chunk ch - 1 has been consumed
      fetch(ch + FW_STAGES - 1);
      const unsigned char* s = smem + (ch % FW_STAGES) * FW_STAGE;
      const unsigned char* ar = s + row * FW_LD;
      const unsigned char* x = s + (FW_ROWS + cg) * FW_LD;
      if (nv == 4) chunk<4>(ar, x, acc);
      else if (nv == 3) chunk<3>(ar, x, acc);
      else if (nv == 2) chunk<2>(ar, x, acc);
      else if (nv == 1) chunk<1>(ar, x, acc);
    }
    __syncthreads();             // before the next columns' first chunks
    if (row0 + row < a.M) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j < nv) {
          const int p = tc::div_rhs(c0 + cg + j, mg), k = c0 + cg + j - p * a.nrhs;
          float2* d = a.dst + ((int64_t)a.pairs[tile.y + p].y * a.nrhs + k) * a.dst_ld + row0 + row;
          tc::red_add2((float*)d, acc[j].x, acc[j].y);
        }
    }
  }
}

}  // namespace

void launch_gemm_stage_few(const GemmArgs& a, LaunchStream s) {
  if (a.ntiles == 0) return;
  if (a.Kd % 8 || a.src_ld % 2) throw Error(-5, "few-column stage needs source ranks that are multiples of 8");
  const dim3 grid((unsigned)a.ntiles, (unsigned)((a.M + FW_ROWS - 1) / FW_ROWS));
  launch_pdl(gemm_few_kernel, grid, FW_THREADS, FW_SMEM, s, a);
  DFMM_CUDA(cudaGetLastError());
}

}  // namespace dfmm
