// Iterative solve around the resident matvec: restarted GMRES for
//
//     (alpha I + beta G) x = b
//
// where G is the plan's operator (Eq. 1).  The paper's method is a fast matvec
// for the iterative solution of integral equations (Sec. 1: each iteration of a
// Krylov method applies G once); this is that outer loop, with the matvec
// through dfmm_apply on the caller's stream.  The Krylov basis lives on the
// device (complex64); each new vector is orthogonalised by classical
// Gram-Schmidt done twice (two kernels per pass, krylov.cu), the small
// Hessenberg least-squares problem is solved on the host in double precision
// with Givens rotations; the host waits once per iteration, and then also sees
// whether a device wait of an apply gave up.
#include <cmath>
#include <complex>
#include <cstring>
#include <string>
#include <vector>

#include "common.h"
#include "dfmm.h"
#include "internal.h"
#include "krylov.h"

namespace {

using cd = std::complex<double>;

struct DevBuf {
  void* p = nullptr;
  ~DevBuf() {
    if (p) cudaFree(p);
  }
};

float2 c32(cd z) { return make_float2((float)z.real(), (float)z.imag()); }

}  // namespace

extern "C" int dfmm_solve(dfmm_plan_t plan, double alpha_re, double alpha_im, double beta_re, double beta_im,
                          const void* b, void* x, int restart, int maxit, double tol, cudaStream_t stream,
                          int* iters, double* relres) {
  try {
    if (!plan || !b || !x) return dfmm::set_error(DFMM_ERR_INVALID, "null argument");
    if (b == x) return dfmm::set_error(DFMM_ERR_INVALID, "b and x must not alias");
    if (restart < 1 || restart > 500) return dfmm::set_error(DFMM_ERR_INVALID, "restart must be in [1, 500]");
    if (maxit < 1) return dfmm::set_error(DFMM_ERR_INVALID, "maxit must be >= 1");
    if (!(tol > 0)) return dfmm::set_error(DFMM_ERR_INVALID, "tol must be positive");
    dfmm_stats st{};
    dfmm_plan_stats(plan, &st);
    if (st.arith != 32) return dfmm::set_error(DFMM_ERR_UNSUPPORTED, "dfmm_solve takes plans that compute in FP32");
    const int64_t N = st.N;
    const int m = restart;
    const cd alpha(alpha_re, alpha_im), beta(beta_re, beta_im);
    // basis, one vector, and beside the kernels' scratch what the host reads back in one copy: the
    // norm of the new vector, the applies' status words so far and the vector's products with the basis
    // in the two passes
    DevBuf Vb, wb, hb;
    const int64_t scratch = (dfmm::krylov_scratch_bytes(N, m + 1) + 255) & ~(int64_t)255;
    constexpr size_t head = 2 * sizeof(double);   // the norm and the status
    const size_t back = head + 2 * (size_t)(m + 1) * sizeof(float2);
    if (dfmm::device_malloc(&Vb.p, (size_t)(m + 1) * N * sizeof(float2)) != cudaSuccess ||
        dfmm::device_malloc(&wb.p, (size_t)N * sizeof(float2)) != cudaSuccess ||
        dfmm::device_malloc(&hb.p, scratch + back) != cudaSuccess) {
      cudaGetLastError();
      return dfmm::set_error(DFMM_ERR_OOM, "GMRES workspace allocation failed");
    }
    DFMM_CUDA(cudaMemsetAsync(hb.p, 0, 256, stream));
    DFMM_CUDA(cudaMemsetAsync((char*)hb.p + scratch, 0, head, stream));
    float2* V = (float2*)Vb.p;
    float2* w = (float2*)wb.p;
    double* nd = (double*)((char*)hb.p + scratch);
    float2* hd = (float2*)((char*)nd + head);
    dfmm::StatusGather gather{nullptr, (unsigned*)(nd + 1)};
    float2* xv = (float2*)x;
    const float2* bv = (const float2*)b;
    const float2 ca = c32(alpha), cb = c32(beta);
    std::vector<char> hback(back);
    auto read_back = [&](size_t bytes) {
      DFMM_CUDA(cudaMemcpyAsync(hback.data(), nd, bytes, cudaMemcpyDeviceToHost, stream));
      DFMM_CUDA(cudaStreamSynchronize(stream));
      unsigned st;
      std::memcpy(&st, hback.data() + sizeof(double), sizeof st);
      if (const int rc = dfmm::status_error(st)) throw dfmm::Error(rc, dfmm_last_error());
      double r;
      std::memcpy(&r, hback.data(), sizeof r);
      return r;
    };

    auto apply = [&](const float2* v, float2* out) {
      const int rc = dfmm_apply(plan, v, out, 1, stream);
      if (rc != DFMM_OK) throw dfmm::Error(rc, dfmm_last_error());
      gather.word = dfmm::apply_status_word(plan, stream);
    };
    auto nrm = [&](float2* v) {
      dfmm::krylov_update(V, 0, nullptr, v, nd, hb.p, N, stream);
      return read_back(head);
    };
    // r = b - A x into dst
    auto residual = [&](float2* dst) {
      apply(xv, w);
      dfmm::krylov_combine(c32(-alpha), xv, c32(-beta), w, make_float2(1.f, 0.f), bv, dst, gather, N,
                           stream);
    };

    const double bnorm = nrm((float2*)bv);   // no columns: only read
    int done = 0;
    double rr = 0.0;
    if (bnorm == 0.0) {
      DFMM_CUDA(cudaMemsetAsync(xv, 0, (size_t)N * sizeof(float2), stream));
    } else {
      std::vector<cd> H((size_t)(m + 1) * m), g(m + 1), cs(m), sn(m), y(m);
      std::vector<float2> yc(m);
      while (done < maxit) {
        residual(V);
        const double beta0 = nrm(V);
        rr = beta0 / bnorm;
        if (rr <= tol) break;
        dfmm::krylov_scale(V, nd, N, stream);
        std::fill(H.begin(), H.end(), cd(0));
        std::fill(g.begin(), g.end(), cd(0));
        g[0] = beta0;
        int k = 0;
        for (int j = 0; j < m && done < maxit; ++j) {
          const float2* v = V + (size_t)j * N;
          float2* vj = V + (size_t)(j + 1) * N;
          // vj = (alpha I + beta G) v, orthogonalised by classical Gram-Schmidt, twice
          apply(v, w);
          dfmm::krylov_dots(V, j + 1, vj, w, cb, v, ca, hd, hb.p, gather, N, stream);
          dfmm::krylov_update(V, j + 1, hd, vj, nd, hb.p, N, stream);
          dfmm::krylov_dots(V, j + 1, vj, nullptr, cb, nullptr, ca, hd + m + 1, hb.p, dfmm::StatusGather{}, N, stream);
          dfmm::krylov_update(V, j + 1, hd + m + 1, vj, nd, hb.p, N, stream);
          dfmm::krylov_scale(vj, nd, N, stream);
          const double hn = read_back(back);
          const float2* hh = (const float2*)(hback.data() + head);
          for (int i = 0; i <= j; ++i)
            H[(size_t)i * m + j] = cd(hh[i].x, hh[i].y) + cd(hh[m + 1 + i].x, hh[m + 1 + i].y);
          H[(size_t)(j + 1) * m + j] = hn;
          // earlier rotations, then a new one that zeroes H[j+1][j]
          for (int i = 0; i < j; ++i) {
            const cd a = H[(size_t)i * m + j], c = H[(size_t)(i + 1) * m + j];
            H[(size_t)i * m + j] = std::conj(cs[i]) * a + std::conj(sn[i]) * c;
            H[(size_t)(i + 1) * m + j] = -sn[i] * a + cs[i] * c;
          }
          const cd a = H[(size_t)j * m + j];
          const double den = std::sqrt(std::norm(a) + hn * hn);
          cs[j] = den > 0 ? a / den : cd(1);
          sn[j] = den > 0 ? cd(hn / den) : cd(0);
          H[(size_t)j * m + j] = den;
          H[(size_t)(j + 1) * m + j] = 0;
          g[j + 1] = -sn[j] * g[j];
          g[j] = std::conj(cs[j]) * g[j];
          ++done;
          k = j + 1;
          rr = std::abs(g[j + 1]) / bnorm;
          if (rr <= tol || hn == 0.0) break;
        }
        // y = H[0:k, 0:k]^-1 g[0:k];  x += V[:, 0:k] y
        for (int i = k - 1; i >= 0; --i) {
          cd s = g[i];
          for (int l = i + 1; l < k; ++l) s -= H[(size_t)i * m + l] * y[l];
          y[i] = s / H[(size_t)i * m + i];
        }
        for (int i = 0; i < k; ++i) yc[i] = c32(-y[i]);
        DFMM_CUDA(cudaMemcpyAsync(hd, yc.data(), (size_t)k * sizeof(float2), cudaMemcpyHostToDevice, stream));
        dfmm::krylov_update(V, k, hd, xv, nd, hb.p, N, stream);
        DFMM_CUDA(cudaStreamSynchronize(stream));
        if (rr <= tol) break;
      }
      // the true residual of the returned x
      residual(V);
      rr = nrm(V) / bnorm;
    }
    DFMM_CUDA(cudaStreamSynchronize(stream));
    if (iters) *iters = done;
    if (relres) *relres = rr;
    return DFMM_OK;
  } catch (const dfmm::Error& e) {
    return dfmm::set_error(e.code, e.what());
  } catch (const std::exception& e) {
    return dfmm::set_error(DFMM_ERR_INVALID, e.what());
  }
}
