// Trailing update on the CUDA cores: C -= A * B (row-major), FP64 (DFMA) or FP32.
//
// This is the paper's "inner" block update (arxiv 2202.13995, section "Base
// Implementation": the inner blocks are updated by matrix multiplication of
// the left and top blocks), A22 <- A22 - L21 * U12.  On GB300 the FP64 rate is
// a small fraction of the FP32 rate and tcgen05 has no FP64 kind, so the FP64
// path is bound by DFMA issue: a 64 x 64 CTA tile with a 4 x 4 register tile
// per thread keeps the FP64 pipes fed from shared memory with ample slack.
#include "common.cuh"
#include "kernels.h"

namespace gb {

constexpr int SG_BM = 64, SG_BN = 64, SG_BK = 16;

template <typename T>
__global__ void __launch_bounds__(256) gemm_simt_kernel(T* __restrict__ C, int64_t ldc, const T* __restrict__ A,
                                                        int64_t lda, const T* __restrict__ B, int64_t ldb, int m,
                                                        int n, int k) {
  __shared__ T As[2][SG_BK][SG_BM];
  __shared__ T Bs[2][SG_BK][SG_BN];
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.y * SG_BM, n0 = blockIdx.x * SG_BN;

  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = T(0);

  T ra[4], rb[4];
  auto load_regs = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int e = tid + 256 * q;
      const int ar = e >> 4, ak = e & 15;
      const int gr = m0 + ar, gk = k0 + ak;
      ra[q] = (gr < m && gk < k) ? A[(int64_t)gr * lda + gk] : T(0);
      const int bk = e >> 6, bc = e & 63;
      const int gbk = k0 + bk, gc = n0 + bc;
      rb[q] = (gbk < k && gc < n) ? B[(int64_t)gbk * ldb + gc] : T(0);
    }
  };
  auto store_smem = [&](int buf) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int e = tid + 256 * q;
      As[buf][e & 15][e >> 4] = ra[q];
      Bs[buf][e >> 6][e & 63] = rb[q];
    }
  };

  const int nk = (k + SG_BK - 1) / SG_BK;
  load_regs(0);
  store_smem(0);
  __syncthreads();
  for (int t = 0; t < nk; ++t) {
    const int buf = t & 1;
    if (t + 1 < nk) load_regs((t + 1) * SG_BK);
#pragma unroll
    for (int kk = 0; kk < SG_BK; ++kk) {
      T a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[buf][kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[buf][kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    if (t + 1 < nk) {
      store_smem(buf ^ 1);
      __syncthreads();
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = m0 + ty + 16 * i;
    if (r >= m) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = n0 + tx + 16 * j;
      if (c < n) C[(int64_t)r * ldc + c] -= acc[i][j];
    }
  }
}

// Small FP64 updates: tiles of BM x 32, BM / 8 elements per thread.  A 64 x 64 tile
// with k = 64 keeps one SM's FP64 pipes for 63 us, so an update of few tiles
// leaves most SMs idle; smaller tiles spread it (launch_gemm_simt chooses).
template <int BM>
__global__ void __launch_bounds__(256) gemm_small_f64_kernel(double* __restrict__ C, int64_t ldc,
                                                             const double* __restrict__ A, int64_t lda,
                                                             const double* __restrict__ B, int64_t ldb, int m, int n,
                                                             int k) {
  constexpr int BN = 32, BK = 32, RI = BM / 8;
  __shared__ double As[BM][BK + 1];
  __shared__ double Bs[BK][BN];
  const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  double acc[RI];
#pragma unroll
  for (int i = 0; i < RI; ++i) acc[i] = 0.0;
  double ra[RI], rb[4];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < RI; ++q) {
      const int r = m0 + ty + 8 * q, c = k0 + tx;
      ra[q] = r < m && c < k ? A[(int64_t)r * lda + c] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = k0 + ty + 8 * q, c = n0 + tx;
      rb[q] = r < k && c < n ? B[(int64_t)r * ldb + c] : 0.0;
    }
  };
  load(0);
  for (int k0 = 0; k0 < k; k0 += BK) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < RI; ++q) As[ty + 8 * q][tx] = ra[q];
#pragma unroll
    for (int q = 0; q < 4; ++q) Bs[ty + 8 * q][tx] = rb[q];
    __syncthreads();
    if (k0 + BK < k) load(k0 + BK);
#pragma unroll 8
    for (int kk = 0; kk < BK; ++kk) {
      const double b = Bs[kk][tx];
#pragma unroll
      for (int i = 0; i < RI; ++i) acc[i] = fma(As[ty + 8 * i][kk], b, acc[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < RI; ++i) {
    const int r = m0 + ty + 8 * i, c = n0 + tx;
    if (r < m && c < n) C[(int64_t)r * ldc + c] -= acc[i];
  }
}

template <typename T>
cudaError_t launch_gemm_simt(T* C, int64_t ldc, const T* A, int64_t lda, const T* B, int64_t ldb, int m, int n,
                             int k, const DevInfo& dev, cudaStream_t st) {
  if (m <= 0 || n <= 0 || k <= 0) return cudaSuccess;
  dim3 grid((unsigned)cdiv(n, SG_BN), (unsigned)cdiv(m, SG_BM));
  if (grid.y > 65535u) return cudaErrorInvalidConfiguration;
  if constexpr (sizeof(T) == 8) {
    // (fewer 64 x 64 tiles than twice the SMs, 304 on GB300, leave their FP64 pipes unevenly
    // loaded: k = 64, us with 64 x 64 tiles and with these: 384 rows 72 and 21, 640
    // 73 and 54, 900 138 and 103, 1100 (324 tiles) 203 and 203)
    const int64_t tiles = (int64_t)grid.x * grid.y;
    const int64_t wave = 2 * dev.sm_count;
    if (tiles < wave) {
      if (cdiv(m, 32) * cdiv(n, 32) >= wave)
        gemm_small_f64_kernel<32><<<dim3((unsigned)cdiv(n, 32), (unsigned)cdiv(m, 32)), 256, 0, st>>>(C, ldc, A, lda, B,
                                                                                                  ldb, m, n, k);
      else
        gemm_small_f64_kernel<8><<<dim3((unsigned)cdiv(n, 32), (unsigned)cdiv(m, 8)), 256, 0, st>>>(C, ldc, A, lda, B,
                                                                                                ldb, m, n, k);
      return cudaGetLastError();
    }
  }
  gemm_simt_kernel<T><<<grid, 256, 0, st>>>(C, ldc, A, lda, B, ldb, m, n, k);
  return cudaGetLastError();
}

// The blocks that a certified split update left alone (gemm_ozaki.cu):
// 32 rows x 64 columns of C -= A B each, 2 x 4 elements per thread, bound by
// FP64 issue like gemm_simt_kernel.  Persistent CTAs walk the list; with none
// listed (the usual case) the launch costs a few microseconds.
constexpr int GL_BM = 32, GL_BN = 64, GL_BK = 32;

__global__ void __launch_bounds__(256) gemm_list_kernel(double* __restrict__ C, int64_t ldc,
                                                        const double* __restrict__ A, int64_t lda,
                                                        const double* __restrict__ B, int64_t ldb, int m, int n, int k,
                                                        int* off, int tag, const int* cnt, const int* list) {
  __shared__ double As[GL_BK][GL_BM + 1];
  __shared__ double Bs[GL_BK][GL_BN];
  const int nbn = (n + GL_BN - 1) / GL_BN;
  const int all = ((m + GL_BM - 1) / GL_BM) * nbn;
  // (raised by an earlier update, never by this launch's own block 0)
  const int raised = __ldcg(off);
  const bool whole = raised != 0 && raised != tag;
  const int count = whole ? all : min(__ldcg(cnt), all);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int it = blockIdx.x; it < count; it += gridDim.x) {
    const int b = whole ? it : list[it];
    const int m0 = (b / nbn) * GL_BM, n0 = (b % nbn) * GL_BN;
    double acc[2][4] = {};
    for (int k0 = 0; k0 < k; k0 += GL_BK) {
      double ra[GL_BM * GL_BK / 256], rb[GL_BN * GL_BK / 256];
#pragma unroll
      for (int q = 0; q < GL_BM * GL_BK / 256; ++q) {
        const int e = tid + 256 * q, r = m0 + e / GL_BK, c = k0 + e % GL_BK;
        ra[q] = r < m && c < k ? A[(int64_t)r * lda + c] : 0.0;
      }
#pragma unroll
      for (int q = 0; q < GL_BN * GL_BK / 256; ++q) {
        const int e = tid + 256 * q, r = k0 + e / GL_BN, c = n0 + e % GL_BN;
        rb[q] = r < k && c < n ? B[(int64_t)r * ldb + c] : 0.0;
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < GL_BM * GL_BK / 256; ++q) {
        const int e = tid + 256 * q;
        As[e % GL_BK][e / GL_BK] = ra[q];
      }
#pragma unroll
      for (int q = 0; q < GL_BN * GL_BK / 256; ++q) {
        const int e = tid + 256 * q;
        Bs[e / GL_BN][e % GL_BN] = rb[q];
      }
      __syncthreads();
#pragma unroll 8
      for (int kk = 0; kk < GL_BK; ++kk) {
        const double a0 = As[kk][ty], a1 = As[kk][ty + 16];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const double bv = Bs[kk][tx + 16 * j];
          acc[0][j] = fma(a0, bv, acc[0][j]);
          acc[1][j] = fma(a1, bv, acc[1][j]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int r = m0 + ty + 16 * i;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = n0 + tx + 16 * j;
        if (r < m && c < n) C[(int64_t)r * ldc + c] -= acc[i][j];
      }
    }
  }
  // (the split update costs about a twentieth of the plain one, so it pays
  // until nearly every block comes here)
  if (blockIdx.x == 0 && tid == 0 && !whole && (int64_t)count * 10 > (int64_t)all * 9) *off = tag;
}

cudaError_t launch_gemm_list(double* C, int64_t ldc, const double* A, int64_t lda, const double* B, int64_t ldb, int m,
                             int n, int k, const OzCert& cert, const DevInfo& dev, cudaStream_t st) {
  if (m <= 0 || n <= 0 || k <= 0) return cudaSuccess;
  const int64_t blocks = (int64_t)oz_cert_blocks(m, n);
  const int grid = (int)(blocks < 4 * dev.sm_count ? blocks : 4 * dev.sm_count);
  gemm_list_kernel<<<grid, 256, 0, st>>>(C, ldc, A, lda, B, ldb, m, n, k, cert.off, cert.tag, cert.cnt, cert.list);
  return cudaGetLastError();
}

template cudaError_t launch_gemm_simt<double>(double*, int64_t, const double*, int64_t, const double*, int64_t, int,
                                              int, int, const DevInfo&, cudaStream_t);
template cudaError_t launch_gemm_simt<float>(float*, int64_t, const float*, int64_t, const float*, int64_t, int, int,
                                             int, const DevInfo&, cudaStream_t);

}  // namespace gb
