// k_lambda.cu -- the dominant contraction of the sweep: lambda products of
// whole orbital rows (Sec. AGP, Eq. agp_expansion), A_up rows phi^T lambda and
// Bt rows lambda phi, batched over walkers.
#include "jagp_group.cuh"
#include "jagp_launch.h"

namespace jagp {

// ---------------------------------------------------------------------------
// lambda products of whole orbital rows, batched over walkers:
//   Out[row][c] = sum_k P[row][k] Lam[k][c]
// with Lam = lambda (A_up rows phi^T lambda) or lambda^T (Bt rows lambda phi).
// In the sweep only the accepted moves' rows are listed, so the cost is
// (accepted moves) x L^2.  T x T output tile, 256 threads each holding an
// (T/16) x (T/16) register block (rows ty + 16 i, columns tx + 16 j), k-chunks
// of 16 (T = 64) or 32.  FP64 CUDA-core arithmetic: a warp's FMA occupies the SM's
// FP64 pipe for 16 clocks, so even one output per thread (two shared-memory
// reads per FMA) is bound by that pipe, and the tile only decides how evenly the
// outputs spread over the SMs and how much of a tile is padding.
// ---------------------------------------------------------------------------
template <int T>
struct LambdaRows {
  static __device__ __forceinline__ void run(const double *__restrict__ P, const double *__restrict__ Lam,
                                             double *__restrict__ Out, const int *__restrict__ list,
                                             const int *__restrict__ count, int nrows, int nsub, int stride, int L,
                                             const uint3 bid, const uint3 gdim) {
    assume_global(P, Lam, Out);
    constexpr int R = T / 16, KC = T == 64 ? 16 : 32;
    const int rows = count ? *count : nrows;
    const int m0 = bid.y * T;
    if (m0 >= rows) return;
    const int n0 = bid.x * T;
    __shared__ double As[KC][T + 1];
    __shared__ double Bs[KC][T];
    __shared__ long rowoff[T];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    if (tid < T) {
      const int m = m0 + tid;
      long phys = -1;
      if (m < rows) phys = list ? (long)list[m] : (long)(m / nsub) * stride + (m % nsub);
      rowoff[tid] = phys < 0 ? -1 : phys * (long)L;
    }
    __syncthreads();
    double acc[R][R];
  #pragma unroll
    for (int i = 0; i < R; ++i)
  #pragma unroll
      for (int j = 0; j < R; ++j) acc[i][j] = 0.0;
    for (int k0 = 0; k0 < L; k0 += KC) {
  #pragma unroll
      for (int q = 0; q < T * KC / 256; ++q) {
        // consecutive threads take consecutive k of a row of P, consecutive columns of a row of Lam
        const int idx = tid + q * 256, ar = idx / KC, ak = idx % KC, bk = idx / T, bc = idx % T;
        const long ro = rowoff[ar];
        As[ak][ar] = (ro >= 0 && k0 + ak < L) ? P[ro + k0 + ak] : 0.0;
        Bs[bk][bc] = (k0 + bk < L && n0 + bc < L) ? Lam[(size_t)(k0 + bk) * L + n0 + bc] : 0.0;
      }
      __syncthreads();
      if (L - k0 >= KC) {
  #pragma unroll
        for (int kk = 0; kk < KC; ++kk) step(As[kk], Bs[kk], tx, ty, acc);
      } else {
        for (int kk = 0; kk < L - k0; ++kk) step(As[kk], Bs[kk], tx, ty, acc);
      }
      __syncthreads();
    }
  #pragma unroll
    for (int i = 0; i < R; ++i) {
      const long ro = rowoff[ty + 16 * i];
      if (ro < 0) continue;
  #pragma unroll
      for (int j = 0; j < R; ++j) {
        const int c = n0 + tx + 16 * j;
        if (c < L) Out[ro + c] = acc[i][j];
      }
    }
}
  static __device__ __forceinline__ void step(const double *a_row, const double *b_row, int tx, int ty,
                                              double (&acc)[T / 16][T / 16]) {
    constexpr int R = T / 16;
    double a[R], b[R];
  #pragma unroll
    for (int i = 0; i < R; ++i) a[i] = a_row[ty + 16 * i];
  #pragma unroll
    for (int j = 0; j < R; ++j) b[j] = b_row[tx + 16 * j];
  #pragma unroll
    for (int i = 0; i < R; ++i)
  #pragma unroll
      for (int j = 0; j < R; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
  }
};
template <int T>
__global__ void __launch_bounds__(256) k_lambda_rows(const double *__restrict__ P, const double *__restrict__ Lam,
                                                     double *__restrict__ Out, const int *__restrict__ list,
                                                     const int *__restrict__ count, int nrows, int nsub, int stride,
                                                     int L) {
  LambdaRows<T>::run(P, Lam, Out, list, count, nrows, nsub, stride, L, blockIdx, gridDim);
}

template <int T>
static cudaError_t launch_tile(const double *P, const double *Lam, double *Out, const int *list, const int *count,
                               int nrows, int nsub, int stride, int L, int max_rows, cudaStream_t st) {
  dim3 grid((L + T - 1) / T, (max_rows + T - 1) / T);
  return launch_or_record<LambdaRows<T>, 256>(k_lambda_rows<T>, grid, dim3(256), 0, st, P, Lam, Out, list, count,
                                              nrows, nsub > 0 ? nsub : 1, stride, L);
}

cudaError_t launch_lambda_rows(const double *P, const double *Lam, double *Out, const int *list, const int *count,
                               int nrows, int nsub, int stride, int L, int max_rows, cudaStream_t st) {
  if (max_rows <= 0) return cudaSuccess;
  // the tile whose fullest SM has the least FP64 work (the sums of an output
  // run over k in the same order in each, so the choice changes no result);
  // the factors are the smaller tiles' extra loads and barriers.  A grouped launch
  // fills the SMs with many systems' tiles: one tile for all, so that they share it.
  if (group_recorder()) return launch_tile<32>(P, Lam, Out, list, count, nrows, nsub, stride, L, max_rows, st);
  auto work = [&](int t, double f) {
    const long long tiles = (long long)((L + t - 1) / t) * ((max_rows + t - 1) / t);
    return f * (double)((tiles + 151) / 152) * t * t;
  };
  const double w64 = work(64, 1.0), w32 = work(32, 1.02), w16 = work(16, 1.08);
  if (w16 < w32 && w16 < w64)
    return launch_tile<16>(P, Lam, Out, list, count, nrows, nsub, stride, L, max_rows, st);
  if (w32 < w64) return launch_tile<32>(P, Lam, Out, list, count, nrows, nsub, stride, L, max_rows, st);
  return launch_tile<64>(P, Lam, Out, list, count, nrows, nsub, stride, L, max_rows, st);
}

}  // namespace jagp
