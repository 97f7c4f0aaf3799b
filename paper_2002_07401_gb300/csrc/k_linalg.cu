// k_linalg.cu -- the dense contractions and the FP64 inverse refresh of the
// geminal matrix (Sec. AGP, Eq. agp_expansion: G~ = Phi_up lambda Phi_dn^T | Phi_up C).
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "jagp_group.cuh"
#include "jagp_launch.h"

namespace jagp {

// ---------------------------------------------------------------------------
// Per-walker small GEMM against row-major operands sharing the contraction
// index:  Out[w][a][b] = sum_k X[w][a][k] Y[w][b][k].
// Used for the proposed rows (Phi'_up . Bt), the proposed columns
// (Phi'_dn . A_up) and G~ at a refresh (Phi_up . Bt).  16 x 16 output tile per
// CTA, one output per thread, operands staged through shared memory in
// k-chunks of 64 (row pitch 65 doubles: conflict-free column reads).
// ---------------------------------------------------------------------------
template <typename T>
struct GemmRows {
  static __device__ __forceinline__ void run(const T *__restrict__ X, size_t xw, const T *__restrict__ Y, size_t yw,
                                             int ma, int nb, int K, T *__restrict__ Out, size_t ow, int ldo,
                                             const uint3 bid, const uint3 gdim) {
    assume_global(X, Y, Out);
    __shared__ T Xs[16][65];
    __shared__ T Ys[16][65];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int w = bid.z, a0 = bid.y * 16, b0 = bid.x * 16;
    const T *Xw = X + (size_t)w * xw;
    const T *Yw = Y + (size_t)w * yw;
    T acc = T(0);
    for (int k0 = 0; k0 < K; k0 += 64) {
  #pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int idx = threadIdx.x + q * 256, row = idx >> 6, col = idx & 63;
        const int k = k0 + col;
        const int a = a0 + row, b = b0 + row;
        Xs[row][col] = (a < ma && k < K) ? Xw[(size_t)a * K + k] : T(0);
        Ys[row][col] = (b < nb && k < K) ? Yw[(size_t)b * K + k] : T(0);
      }
      __syncthreads();
  #pragma unroll 16
      for (int k = 0; k < 64; ++k) acc = fma(Xs[ty][k], Ys[tx][k], acc);
      __syncthreads();
    }
    if (a0 + ty < ma && b0 + tx < nb) Out[(size_t)w * ow + (size_t)(a0 + ty) * ldo + b0 + tx] = acc;
}
};
template <typename T>
__global__ void __launch_bounds__(256) k_gemm_rows(const T *__restrict__ X, size_t xw, const T *__restrict__ Y,
                                                   size_t yw, int ma, int nb, int K, T *__restrict__ Out, size_t ow,
                                                   int ldo) {
  GemmRows<T>::run(X, xw, Y, yw, ma, nb, K, Out, ow, ldo, blockIdx, gridDim);
}

// The same products for ma, nb <= NB = 2, 4 or 8: 256 / NB^2 walkers per CTA,
// one output per thread (a 16 x 16 tile of one walker would be mostly padding:
// 2 x 2 outputs used 1.6 % of it).  The sum over k keeps its order.
template <typename T, int NB>
struct GemmRowsTiny {
  static __device__ __forceinline__ void run(const T *__restrict__ X, size_t xw, const T *__restrict__ Y, size_t yw,
                                             int ma, int nb, int K, T *__restrict__ Out, size_t ow, int ldo, int W,
                                             const uint3 bid, const uint3 gdim) {
    assume_global(X, Y, Out);
    constexpr int WK = 256 / (NB * NB), KC = 16, ROWS = WK * NB;  // walkers per CTA, staged rows per operand
    __shared__ T Xs[ROWS][KC + 1];
    __shared__ T Ys[ROWS][KC + 1];
    const int tid = threadIdx.x, wl = tid / (NB * NB), a = tid / NB % NB, b = tid % NB;
    const int w0 = bid.x * WK, w = w0 + wl;
    T acc = T(0);
    for (int k0 = 0; k0 < K; k0 += KC) {
      for (int idx = tid; idx < ROWS * KC; idx += 256) {
        const int row = idx / KC, kk = idx % KC, wr = w0 + row / NB, i = row % NB, k = k0 + kk;
        const bool in = wr < W && k < K;
        Xs[row][kk] = in && i < ma ? X[(size_t)wr * xw + (size_t)i * K + k] : T(0);
        Ys[row][kk] = in && i < nb ? Y[(size_t)wr * yw + (size_t)i * K + k] : T(0);
      }
      __syncthreads();
  #pragma unroll
      for (int kk = 0; kk < KC; ++kk) acc = fma(Xs[wl * NB + a][kk], Ys[wl * NB + b][kk], acc);
      __syncthreads();
    }
    if (w < W && a < ma && b < nb) Out[(size_t)w * ow + (size_t)a * ldo + b] = acc;
}
};
template <typename T, int NB>
__global__ void __launch_bounds__(256) k_gemm_rows_tiny(const T *__restrict__ X, size_t xw, const T *__restrict__ Y,
                                                        size_t yw, int ma, int nb, int K, T *__restrict__ Out,
                                                        size_t ow, int ldo, int W) {
  GemmRowsTiny<T, NB>::run(X, xw, Y, yw, ma, nb, K, Out, ow, ldo, W, blockIdx, gridDim);
}

// The FP32 path's per-walker products of up to 32 rows (the proposed rows and
// columns, plain; the refresh's G~ = Phi_up Bt^T, DOT2): 4 x 4 outputs per
// thread, Q x Q threads per walker (Q = ceil(rows / 4)), as many walkers as fill
// 128 threads; operands through shared memory in k-chunks of 16, transposed, so
// that sixteen outputs take two 16-byte reads per term (one output per thread was
// bound by its two or four reads), the next chunk loading into registers
// meanwhile.  Every output sums over k in order.
// DOT2: a compensated dot product (error-free product by fma, error-free sum,
// the errors summed separately; Ogita, Rump and Oishi 2005) over two-float
// operands X + Xlo and Y + Ylo (the low parts' products with the high parts go
// into the error sum; lo * lo is below the result's precision), so that G~ is
// as accurate as the double-word tables rather than FP32, kept in FP64.  The _rn
// intrinsics keep the compiler from fusing the steps.
// Plain, 4096 walkers of 16 x 16, K = 320: 107 us with one output per thread, this 46.
// DOT2, 1021 walkers of 24 x 24, K = 460: 324 us with one output per thread, this 203
// (its FP32 instructions alone: 94); up to 16 rows the 2 x 2 kernel below, whose
// fewer registers keep more warps, is as fast (204 us for 4096 walkers of 16 x 16,
// K = 320, against 220).
constexpr int kSmallKC = 16, kSmallThreads = 128;
constexpr int small_walkers(int q) { return q == 1 ? 32 : (q == 2 ? 16 : kSmallThreads / (q * q)); }
constexpr int small_pitch(int q) { return 4 * q + 4; }  // floats per staged k: the transposing stores spread over banks

template <bool DOT2, int Q>
struct GemmSmallF32 {
  using OutT = std::conditional_t<DOT2, double, float>;
  static __device__ __forceinline__ void run(const float *__restrict__ X, const float *__restrict__ Xlo, size_t xw,
                                             const float *__restrict__ Y, const float *__restrict__ Ylo, size_t yw,
                                             int ma, int nb, int K, OutT *__restrict__ Out, size_t ow, int ldo, int W,
                                             int vec, const uint3 bid, const uint3 gdim) {
    assume_global(X, Y, Out);
    extern __shared__ float4 smf4[];
    constexpr int KC = kSmallKC, kOps = DOT2 ? 4 : 2, rows = 4 * Q, wpc = small_walkers(Q), P = small_pitch(Q);
    constexpr int per = kOps * KC * P;  // floats per walker: X, Y (and their low parts), each [KC][P]
    constexpr int kQuads = wpc * kOps * rows * (KC / 4), kLoads = (kQuads + kSmallThreads - 1) / kSmallThreads;
    const int tid = threadIdx.x;
    float *sm = reinterpret_cast<float *>(smf4);
    const int wl = tid / (Q * Q), t = tid - wl * Q * Q, ty = t / Q, tx = t - ty * Q;
    const int w0 = (int)bid.x * wpc, w = w0 + wl;
    const bool active = wl < wpc && w < W;  // idle threads still load and take part in the barriers
    float acc[4][4], cmp[DOT2 ? 4 : 1][DOT2 ? 4 : 1];
  #pragma unroll
    for (int i = 0; i < 4; ++i)
  #pragma unroll
      for (int j = 0; j < 4; ++j) {
        acc[i][j] = 0.0f;
        if constexpr (DOT2) cmp[i][j] = 0.0f;
      }
    // quad idx: four consecutive k of one row; consecutive threads take a row's quads
    auto fetch = [&](int idx, int k0) {
      const int k = k0 + 4 * (idx % (KC / 4)), row = idx / (KC / 4) % rows, op = idx / (KC / 4 * rows) % kOps,
                wr = idx / (KC / 4 * rows * kOps);
      const bool y = op & 1;
      const float *src = op >= 2 ? (y ? Ylo : Xlo) : (y ? Y : X);
      float4 f = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (idx < kQuads && w0 + wr < W && row < (y ? nb : ma) && src) {
        const float *g = src + (size_t)(w0 + wr) * (y ? yw : xw) + (size_t)row * K + k;
        if (vec) {  // (K % 4 = 0: a quad is whole or absent)
          if (k < K) f = *reinterpret_cast<const float4 *>(g);
        } else {
          if (k < K) f.x = g[0];
          if (k + 1 < K) f.y = g[1];
          if (k + 2 < K) f.z = g[2];
          if (k + 3 < K) f.w = g[3];
        }
      }
      return f;
    };
    auto put = [&](int idx, const float4 f) {
      const int k4 = idx % (KC / 4), row = idx / (KC / 4) % rows, op = idx / (KC / 4 * rows) % kOps,
                wr = idx / (KC / 4 * rows * kOps);
      if (idx < kQuads) {
        float *d = sm + wr * per + (op * KC + 4 * k4) * P + row;
        d[0] = f.x;
        d[P] = f.y;
        d[2 * P] = f.z;
        d[3 * P] = f.w;
      }
    };
    float4 pre[kLoads];
  #pragma unroll
    for (int l = 0; l < kLoads; ++l) pre[l] = fetch(tid + l * kSmallThreads, 0);
    const float *xs = sm + wl * per + 4 * ty, *ys = sm + wl * per + KC * P + 4 * tx;
    for (int k0 = 0; k0 < K; k0 += KC) {
  #pragma unroll
      for (int l = 0; l < kLoads; ++l) put(tid + l * kSmallThreads, pre[l]);
      __syncthreads();
      if (k0 + KC < K) {
  #pragma unroll
        for (int l = 0; l < kLoads; ++l) pre[l] = fetch(tid + l * kSmallThreads, k0 + KC);
      }
      if (active) {
  #pragma unroll 4
        for (int kk = 0; kk < KC; ++kk) {
          const float4 xv = *reinterpret_cast<const float4 *>(xs + kk * P);
          const float4 yv = *reinterpret_cast<const float4 *>(ys + kk * P);
          const float xa[4] = {xv.x, xv.y, xv.z, xv.w}, yb[4] = {yv.x, yv.y, yv.z, yv.w};
          if constexpr (DOT2) {
            const float4 xw4 = *reinterpret_cast<const float4 *>(xs + (2 * KC + kk) * P);
            const float4 yw4 = *reinterpret_cast<const float4 *>(ys + (2 * KC + kk) * P);
            const float xl[4] = {xw4.x, xw4.y, xw4.z, xw4.w}, yl[4] = {yw4.x, yw4.y, yw4.z, yw4.w};
  #pragma unroll
            for (int i = 0; i < 4; ++i)
  #pragma unroll
              for (int j = 0; j < 4; ++j) {
                const float x = xa[i], y = yb[j], sv = acc[i][j];
                const float p = __fmul_rn(x, y);
                const float pe = __fmaf_rn(x, y, -p);
                const float tt = __fadd_rn(sv, p);
                const float z = __fsub_rn(tt, sv);
                const float se = __fadd_rn(__fsub_rn(sv, __fsub_rn(tt, z)), __fsub_rn(p, z));
                acc[i][j] = tt;
                const float cross = __fmaf_rn(xl[i], y, __fmul_rn(x, yl[j]));
                cmp[i][j] = __fadd_rn(cmp[i][j], __fadd_rn(__fadd_rn(cross, pe), se));
              }
          } else {
  #pragma unroll
            for (int i = 0; i < 4; ++i)
  #pragma unroll
              for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(xa[i], yb[j], acc[i][j]);
          }
        }
      }
      __syncthreads();
    }
    if (!active) return;
  #pragma unroll
    for (int i = 0; i < 4; ++i)
  #pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int a = 4 * ty + i, b = 4 * tx + j;
        if (a >= ma || b >= nb) continue;
        // DOT2: the pair (s, c) carries more than FP32 precision: keep it in FP64
        if constexpr (DOT2)
          Out[(size_t)w * ow + (size_t)a * ldo + b] = static_cast<double>(acc[i][j]) + static_cast<double>(cmp[i][j]);
        else
          Out[(size_t)w * ow + (size_t)a * ldo + b] = acc[i][j];
      }
}
};
template <bool DOT2, int Q>
__global__ void __launch_bounds__(kSmallThreads) k_gemm_small_f32(const float *__restrict__ X, const float *__restrict__ Xlo,
                                                        size_t xw, const float *__restrict__ Y,
                                                        const float *__restrict__ Ylo, size_t yw, int ma, int nb,
                                                        int K, typename GemmSmallF32<DOT2, Q>::OutT *__restrict__ Out,
                                                        size_t ow, int ldo, int W, int vec) {
  GemmSmallF32<DOT2, Q>::run(X, Xlo, xw, Y, Ylo, yw, ma, nb, K, Out, ow, ldo, W, vec, blockIdx, gridDim);
}
// threads per side of a walker's tile; grouped launches take two sizes, so that
// systems share a launch
static int small_q(int ma, int nb) {
  const int q = (std::max(ma, nb) + 3) / 4;
  return group_recorder() ? (q <= 4 ? 4 : 8) : q;
}
template <bool DOT2, int Q>
static cudaError_t launch_small_f32(int q, const float *X, const float *Xlo, size_t xw, const float *Y,
                                    const float *Ylo, size_t yw, int ma, int nb, int K,
                                    typename GemmSmallF32<DOT2, Q>::OutT *Out, size_t ow, int ldo, int W,
                                    cudaStream_t st) {
  if constexpr (Q > (DOT2 ? 5 : 1))  // (DOT2: more than 16 rows)
    if (q < Q) return launch_small_f32<DOT2, Q - 1>(q, X, Xlo, xw, Y, Ylo, yw, ma, nb, K, Out, ow, ldo, W, st);
  constexpr int wpc = small_walkers(Q);
  // 16-byte loads along k where every row starts on 16 bytes
  const uintptr_t at = reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y) |
                       reinterpret_cast<uintptr_t>(Xlo) | reinterpret_cast<uintptr_t>(Ylo);
  const int vec = at % 16 == 0 && K % 4 == 0 && xw % 4 == 0 && yw % 4 == 0;
  const size_t smem = (size_t)wpc * (DOT2 ? 4 : 2) * kSmallKC * small_pitch(Q) * sizeof(float);
  return launch_or_record<GemmSmallF32<DOT2, Q>, kSmallThreads>(k_gemm_small_f32<DOT2, Q>, dim3((W + wpc - 1) / wpc),
                                                                dim3(kSmallThreads), smem, st, X, Xlo, xw, Y, Ylo, yw, ma, nb, K, Out, ow, ldo, W,
                                                      vec);
}

// The FP32 path's plain per-walker products of more than 32 rows: 64 x 64 output
// tile, 64 threads with 8 x 8 outputs each (columns 4 tx .. + 3 and 32 + 4 tx .. + 3, rows
// likewise), k-chunks of 16 with the next chunk loading into registers meanwhile: 64 FMAs per four 16-byte
// reads.  64 walkers, 256 x 256, K = 4096: 1.08 ms (1.53 with 4 x 4 outputs per
// thread and scalar reads).
struct GemmTile64F32 {
  static __device__ __forceinline__ void run(const float *__restrict__ X, size_t xw, const float *__restrict__ Y,
                                             size_t yw, int ma, int nb, int K, float *__restrict__ Out, size_t ow,
                                             int ldo, int vec, const uint3 bid, const uint3 gdim) {
    assume_global(X, Y, Out);
    constexpr int KC = 16, P = 68;
    __shared__ __align__(16) float Xs[KC][P];
    __shared__ __align__(16) float Ys[KC][P];
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const int w = bid.z, a0 = bid.y * 64, b0 = bid.x * 64;
    const bool xin = a0 + tid < ma, yin = b0 + tid < nb;  // this thread's row of each operand
    const float *xr = X + (size_t)w * xw + (size_t)(a0 + tid) * K, *yr = Y + (size_t)w * yw + (size_t)(b0 + tid) * K;
    auto load = [&](const float *row, bool in, int k0, float v[KC]) {
  #pragma unroll
      for (int c = 0; c < KC; c += 4) {
        if (in && vec && k0 + c + 4 <= K) {
          const float4 f = *reinterpret_cast<const float4 *>(row + k0 + c);
          v[c] = f.x;
          v[c + 1] = f.y;
          v[c + 2] = f.z;
          v[c + 3] = f.w;
        } else {
  #pragma unroll
          for (int i = 0; i < 4; ++i) v[c + i] = in && k0 + c + i < K ? row[k0 + c + i] : 0.0f;
        }
      }
    };
    float acc[8][8];
  #pragma unroll
    for (int i = 0; i < 8; ++i)
  #pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = 0.0f;
    float xv[KC], yv[KC];
    load(xr, xin, 0, xv);
    load(yr, yin, 0, yv);
    for (int k0 = 0; k0 < K; k0 += KC) {
  #pragma unroll
      for (int c = 0; c < KC; ++c) {
        Xs[c][tid] = xv[c];
        Ys[c][tid] = yv[c];
      }
      __syncthreads();
      if (k0 + KC < K) {
        load(xr, xin, k0 + KC, xv);
        load(yr, yin, k0 + KC, yv);
      }
  #pragma unroll
      for (int kk = 0; kk < KC; ++kk) {
        const float4 x0 = *reinterpret_cast<const float4 *>(&Xs[kk][4 * ty]);
        const float4 x1 = *reinterpret_cast<const float4 *>(&Xs[kk][32 + 4 * ty]);
        const float4 y0 = *reinterpret_cast<const float4 *>(&Ys[kk][4 * tx]);
        const float4 y1 = *reinterpret_cast<const float4 *>(&Ys[kk][32 + 4 * tx]);
        const float xa[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
        const float yb[8] = {y0.x, y0.y, y0.z, y0.w, y1.x, y1.y, y1.z, y1.w};
  #pragma unroll
        for (int i = 0; i < 8; ++i)
  #pragma unroll
          for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(xa[i], yb[j], acc[i][j]);
      }
      __syncthreads();
    }
  #pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int a = a0 + (i < 4 ? 4 * ty + i : 28 + 4 * ty + i);
      if (a >= ma) continue;
      float *o = Out + (size_t)w * ow + (size_t)a * ldo;
  #pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int b = b0 + (j < 4 ? 4 * tx + j : 28 + 4 * tx + j);
        if (b < nb) o[b] = acc[i][j];
      }
    }
}
};
__global__ void __launch_bounds__(64) k_gemm_tile64_f32(const float *__restrict__ X, size_t xw,
                                                        const float *__restrict__ Y, size_t yw, int ma, int nb, int K,
                                                        float *__restrict__ Out, size_t ow, int ldo, int vec) {
  GemmTile64F32::run(X, xw, Y, yw, ma, nb, K, Out, ow, ldo, vec, blockIdx, gridDim);
}

// ---------------------------------------------------------------------------
// Register-blocked variant for N_up >= 32 (FP64; compensated FP32): a TM x TM
// output tile per CTA of 256 threads, R x R outputs per thread (R = TM / 16),
// operands staged through shared memory in k-chunks of 32, transposed so that
// each thread reads R consecutive entries of a column.  With DOT2 every output
// keeps the compensated pair (s, c) of the kernel above; the order of the
// k-sum is the same as there.
// ---------------------------------------------------------------------------
template <typename T, int TM, bool DOT2, typename OutT>
struct GemmRowsBlk {
  static __device__ __forceinline__ void run(const T *__restrict__ X, const float *__restrict__ Xlo, size_t xw,
                                             const T *__restrict__ Y, const float *__restrict__ Ylo, size_t yw,
                                             int ma, int nb, int K, OutT *__restrict__ Out, size_t ow, int ldo,
                                             const uint3 bid, const uint3 gdim) {
    assume_global(X, Y, Out);
    constexpr int KC = 32, R = TM / 16, PAD = TM + 1;
    __shared__ T Xs[KC][PAD];
    __shared__ T Ys[KC][PAD];
    __shared__ float Xl[DOT2 ? KC : 1][DOT2 ? PAD : 1];
    __shared__ float Yl[DOT2 ? KC : 1][DOT2 ? PAD : 1];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int w = bid.z, a0 = bid.y * TM, b0 = bid.x * TM;
    const T *Xw = X + (size_t)w * xw;
    const T *Yw = Y + (size_t)w * yw;
    T acc[R][R];
    float cmp[DOT2 ? R : 1][DOT2 ? R : 1];
  #pragma unroll
    for (int i = 0; i < R; ++i)
  #pragma unroll
      for (int j = 0; j < R; ++j) {
        acc[i][j] = T(0);
        if constexpr (DOT2) cmp[i][j] = 0.0f;
      }
    for (int k0 = 0; k0 < K; k0 += KC) {
      // TM rows x KC columns of each operand; consecutive threads take consecutive k
  #pragma unroll
      for (int q = 0; q < TM * KC / 256; ++q) {
        const int idx = tid + q * 256, row = idx / KC, kk = idx % KC;
        const int k = k0 + kk, a = a0 + row, b = b0 + row;
        const bool xa = a < ma && k < K, yb = b < nb && k < K;
        const size_t xi = (size_t)a * K + k, yi = (size_t)b * K + k;
        Xs[kk][row] = xa ? Xw[xi] : T(0);
        Ys[kk][row] = yb ? Yw[yi] : T(0);
        if constexpr (DOT2) {
          Xl[kk][row] = (Xlo && xa) ? Xlo[(size_t)w * xw + xi] : 0.0f;
          Yl[kk][row] = (Ylo && yb) ? Ylo[(size_t)w * yw + yi] : 0.0f;
        }
      }
      __syncthreads();
  #pragma unroll 4
      for (int kk = 0; kk < KC; ++kk) {
        T xa[R], yb[R];
  #pragma unroll
        for (int i = 0; i < R; ++i) xa[i] = Xs[kk][ty * R + i];
  #pragma unroll
        for (int j = 0; j < R; ++j) yb[j] = Ys[kk][tx * R + j];
        if constexpr (DOT2) {
          float xl[R], yl[R];
  #pragma unroll
          for (int i = 0; i < R; ++i) xl[i] = Xl[kk][ty * R + i];
  #pragma unroll
          for (int j = 0; j < R; ++j) yl[j] = Yl[kk][tx * R + j];
  #pragma unroll
          for (int i = 0; i < R; ++i)
  #pragma unroll
            for (int j = 0; j < R; ++j) {
              const float x = xa[i], y = yb[j], s = acc[i][j];
              const float p = __fmul_rn(x, y);
              const float pe = __fmaf_rn(x, y, -p);
              const float t = __fadd_rn(s, p);
              const float z = __fsub_rn(t, s);
              const float se = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
              acc[i][j] = t;
              const float cross = __fmaf_rn(xl[i], y, __fmul_rn(x, yl[j]));
              cmp[i][j] = __fadd_rn(cmp[i][j], __fadd_rn(__fadd_rn(cross, pe), se));
            }
        } else {
  #pragma unroll
          for (int i = 0; i < R; ++i)
  #pragma unroll
            for (int j = 0; j < R; ++j) acc[i][j] = fma(xa[i], yb[j], acc[i][j]);
        }
      }
      __syncthreads();
    }
  #pragma unroll
    for (int i = 0; i < R; ++i) {
      const int a = a0 + ty * R + i;
      if (a >= ma) continue;
  #pragma unroll
      for (int j = 0; j < R; ++j) {
        const int b = b0 + tx * R + j;
        if (b >= nb) continue;
        OutT v;
        if constexpr (DOT2)
          v = static_cast<double>(acc[i][j]) + static_cast<double>(cmp[i][j]);
        else
          v = acc[i][j];
        Out[(size_t)w * ow + (size_t)a * ldo + b] = v;
      }
    }
}
};
template <typename T, int TM, bool DOT2, typename OutT>
__global__ void __launch_bounds__(256) k_gemm_rows_blk(const T *__restrict__ X, const float *__restrict__ Xlo,
                                                       size_t xw, const T *__restrict__ Y,
                                                       const float *__restrict__ Ylo, size_t yw, int ma, int nb,
                                                       int K, OutT *__restrict__ Out, size_t ow, int ldo) {
  GemmRowsBlk<T, TM, DOT2, OutT>::run(X, Xlo, xw, Y, Ylo, yw, ma, nb, K, Out, ow, ldo, blockIdx, gridDim);
}

// tile of the blocked variant for an ma x nb output (0: the one-output-per-thread kernel)
inline int gemm_rows_tile(int ma, int nb) {
  const int m = ma < nb ? ma : nb;
  return m >= 64 ? 64 : (m >= 32 ? 32 : 0);
}

// The compensated product for small blocks (ma, nb <= 16): four walkers per
// CTA, 64 threads each with a 2 x 2 output block, so that every shared-memory
// operand read serves two outputs instead of one; k order as above.
struct GemmRowsDot2Small {
  static __device__ __forceinline__ void run(const float *__restrict__ X, const float *__restrict__ Xlo, size_t xw,
                                             const float *__restrict__ Y, const float *__restrict__ Ylo, size_t yw,
                                             int ma, int nb, int K, double *__restrict__ Out, size_t ow, int ldo,
                                             int W, const uint3 bid, const uint3 gdim) {
    assume_global(X, Y, Out);
    constexpr int KC = 32;
    __shared__ float Xs[4][KC][17], Xl[4][KC][17], Ys[4][KC][17], Yl[4][KC][17];
    const int sub = threadIdx.x >> 6, t = threadIdx.x & 63;
    const int w = bid.x * 4 + sub;
    const bool active = w < W;  // inactive groups still take part in the barriers
    const int tx = t & 7, ty = t >> 3;  // outputs (2 ty + i, 2 tx + j)
    float s[2][2] = {{0.0f, 0.0f}, {0.0f, 0.0f}}, c[2][2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
    for (int k0 = 0; k0 < K; k0 += KC) {
      for (int idx = t; idx < 16 * KC; idx += 64) {
        const int row = idx / KC, kk = idx % KC, k = k0 + kk;
        const bool xa = active && row < ma && k < K, yb = active && row < nb && k < K;
        const size_t xi = (size_t)w * xw + (size_t)row * K + k, yi = (size_t)w * yw + (size_t)row * K + k;
        Xs[sub][kk][row] = xa ? X[xi] : 0.0f;
        Xl[sub][kk][row] = (Xlo && xa) ? Xlo[xi] : 0.0f;
        Ys[sub][kk][row] = yb ? Y[yi] : 0.0f;
        Yl[sub][kk][row] = (Ylo && yb) ? Ylo[yi] : 0.0f;
      }
      __syncthreads();
  #pragma unroll 4
      for (int kk = 0; kk < KC; ++kk) {
        const float x0 = Xs[sub][kk][2 * ty], x1 = Xs[sub][kk][2 * ty + 1];
        const float l0 = Xl[sub][kk][2 * ty], l1 = Xl[sub][kk][2 * ty + 1];
        const float y0 = Ys[sub][kk][2 * tx], y1 = Ys[sub][kk][2 * tx + 1];
        const float m0 = Yl[sub][kk][2 * tx], m1 = Yl[sub][kk][2 * tx + 1];
        const float xv[2] = {x0, x1}, xl[2] = {l0, l1}, yv[2] = {y0, y1}, yl[2] = {m0, m1};
  #pragma unroll
        for (int i = 0; i < 2; ++i)
  #pragma unroll
          for (int j = 0; j < 2; ++j) {
            const float x = xv[i], y = yv[j], sv = s[i][j];
            const float p = __fmul_rn(x, y);
            const float pe = __fmaf_rn(x, y, -p);
            const float tt = __fadd_rn(sv, p);
            const float z = __fsub_rn(tt, sv);
            const float se = __fadd_rn(__fsub_rn(sv, __fsub_rn(tt, z)), __fsub_rn(p, z));
            s[i][j] = tt;
            const float cross = __fmaf_rn(xl[i], y, __fmul_rn(x, yl[j]));
            c[i][j] = __fadd_rn(c[i][j], __fadd_rn(__fadd_rn(cross, pe), se));
          }
      }
      __syncthreads();
    }
    if (!active) return;
  #pragma unroll
    for (int i = 0; i < 2; ++i)
  #pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int a = 2 * ty + i, b = 2 * tx + j;
        if (a < ma && b < nb)
          Out[(size_t)w * ow + (size_t)a * ldo + b] = static_cast<double>(s[i][j]) + static_cast<double>(c[i][j]);
      }
}
};
__global__ void __launch_bounds__(256) k_gemm_rows_dot2_small(const float *__restrict__ X,
                                                              const float *__restrict__ Xlo, size_t xw,
                                                              const float *__restrict__ Y,
                                                              const float *__restrict__ Ylo, size_t yw, int ma,
                                                              int nb, int K, double *__restrict__ Out, size_t ow,
                                                              int ldo, int W) {
  GemmRowsDot2Small::run(X, Xlo, xw, Y, Ylo, yw, ma, nb, K, Out, ow, ldo, W, blockIdx, gridDim);
}

cudaError_t launch_gemm_rows_dot2(const float *X, const float *Xlo, size_t xw, const float *Y, const float *Ylo,
                                  size_t yw, int ma, int nb, int K, double *Out, size_t ow, int ldo, int W,
                                  cudaStream_t st, int tile) {
  if (W <= 0 || ma <= 0 || nb <= 0) return cudaSuccess;
  if (tile != -1 && tile != 0 && tile != 16 && tile != 32 && tile != 64) return cudaErrorInvalidValue;
  if (tile == 16 && (ma > 16 || nb > 16)) return cudaErrorInvalidValue;
  // one kernel per size up to 32 rows, whatever the tile asked for; above: blocked tiles
  if (ma <= 16 && nb <= 16)
    return launch_or_record<GemmRowsDot2Small, 256>(k_gemm_rows_dot2_small, dim3((W + 3) / 4), dim3(256), 0, st, X,
                                                     Xlo, xw, Y, Ylo, yw, ma, nb, K, Out, ow, ldo, W);
  if (ma <= 32 && nb <= 32)
    return launch_small_f32<true, 8>(small_q(ma, nb), X, Xlo, xw, Y, Ylo, yw, ma, nb, K, Out, ow, ldo, W, st);
  const int tm = tile == 32 || tile == 64 ? tile : (ma >= 64 && nb >= 64 ? 64 : 32);
  dim3 grid((nb + tm - 1) / tm, (ma + tm - 1) / tm, W);
  if (tm == 64)
    return launch_or_record<GemmRowsBlk<float, 64, true, double>, 256>(k_gemm_rows_blk<float, 64, true, double>, grid,
                                                                       dim3(256), 0, st, X, Xlo, xw, Y, Ylo, yw, ma,
                                                                       nb, K, Out, ow, ldo);
  return launch_or_record<GemmRowsBlk<float, 32, true, double>, 256>(k_gemm_rows_blk<float, 32, true, double>, grid,
                                                                     dim3(256), 0, st, X, Xlo, xw, Y, Ylo, yw, ma, nb,
                                                                     K, Out, ow, ldo);
}

template <typename T>
cudaError_t launch_gemm_rows(const T *X, size_t xw, const T *Y, size_t yw, int ma, int nb, int K, T *Out, size_t ow,
                             int ldo, int W, cudaStream_t st, int tile) {
  if (W <= 0 || ma <= 0 || nb <= 0) return cudaSuccess;
  if (tile != -1 && tile != 0 && tile != 32 && tile != 64) return cudaErrorInvalidValue;
  if constexpr (std::is_same<T, float>::value) {
    // one kernel per size, whatever the tile asked for
    const float *none = nullptr;
    if (ma <= 32 && nb <= 32) 
      return launch_small_f32<false, 8>(small_q(ma, nb), X, none, xw, Y, none, yw, ma, nb, K, Out, ow, ldo, W,
                                        st);
    const int vec = (reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) % 16 == 0 && K % 4 == 0 &&
                    xw % 4 == 0 && yw % 4 == 0;
    return launch_or_record<GemmTile64F32, 64>(k_gemm_tile64_f32, dim3((nb + 63) / 64, (ma + 63) / 64, W), dim3(64), 0,
                                               st, X, xw, Y, yw, ma, nb, K, Out, ow, ldo, vec);
  } else {
  const int tm = tile >= 0 ? tile : gemm_rows_tile(ma, nb);
  if (tm) {
    dim3 grid((nb + tm - 1) / tm, (ma + tm - 1) / tm, W);
    const float *none = nullptr;
    if (tm == 64)
      return launch_or_record<GemmRowsBlk<T, 64, false, T>, 256>(k_gemm_rows_blk<T, 64, false, T>, grid, dim3(256), 0,
                                                                 st, X, none, xw, Y, none, yw, ma, nb, K, Out, ow, ldo);
    return launch_or_record<GemmRowsBlk<T, 32, false, T>, 256>(k_gemm_rows_blk<T, 32, false, T>, grid, dim3(256), 0,
                                                               st, X, none, xw, Y, none, yw, ma, nb, K, Out, ow, ldo);
  }
  const int m = ma > nb ? ma : nb;
  if (m <= 2)
    return launch_or_record<GemmRowsTiny<T, 2>, 256>(k_gemm_rows_tiny<T, 2>, dim3((W + 63) / 64), dim3(256), 0, st, X,
                                                     xw, Y, yw, ma, nb, K, Out, ow, ldo, W);
  if (m <= 4)
    return launch_or_record<GemmRowsTiny<T, 4>, 256>(k_gemm_rows_tiny<T, 4>, dim3((W + 15) / 16), dim3(256), 0, st, X,
                                                     xw, Y, yw, ma, nb, K, Out, ow, ldo, W);
  if (m <= 8)
    return launch_or_record<GemmRowsTiny<T, 8>, 256>(k_gemm_rows_tiny<T, 8>, dim3((W + 3) / 4), dim3(256), 0, st, X,
                                                     xw, Y, yw, ma, nb, K, Out, ow, ldo, W);
  dim3 grid((nb + 15) / 16, (ma + 15) / 16, W);
  return launch_or_record<GemmRows<T>, 256>(k_gemm_rows<T>, grid, dim3(256), 0, st, X, xw, Y, yw, ma, nb, K, Out, ow,
                                            ldo);
  }
}
template cudaError_t launch_gemm_rows<double>(const double *, size_t, const double *, size_t, int, int, int, double *,
                                              size_t, int, int, cudaStream_t, int);
template cudaError_t launch_gemm_rows<float>(const float *, size_t, const float *, size_t, int, int, int, float *,
                                             size_t, int, int, cudaStream_t, int);

template <typename T>
__global__ void k_fill_unpaired(const double *__restrict__ unp, T *__restrict__ bt, int W, int nu, int nd,
                                int L) {
  const int k = nu - nd;
  const long total = (long)W * k * L;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
    const int c = (int)(idx % L);
    const long t = idx / L;
    const int l = (int)(t % k);
    const int w = (int)(t / k);
    bt[((size_t)w * nu + nd + l) * L + c] = static_cast<T>(unp[(size_t)l * L + c]);
  }
}

template <typename T>
cudaError_t launch_fill_unpaired(const DevSystem &s, T *bt, int W, cudaStream_t st) {
  if (W <= 0 || s.n_up == s.n_dn) return cudaSuccess;
  const long total = (long)W * (s.n_up - s.n_dn) * s.L;
  long blocks = (total + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  k_fill_unpaired<T><<<(int)blocks, 256, 0, st>>>(s.unpaired, bt, W, s.n_up, s.n_dn, s.L);
  return cudaGetLastError();
}
template cudaError_t launch_fill_unpaired<double>(const DevSystem &, double *, int, cudaStream_t);

__global__ void k_fill_unpaired_lo(const double *__restrict__ unp, float *__restrict__ lo, int W, int nu, int nd,
                                   int L) {
  const int k = nu - nd;
  const long total = (long)W * k * L;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
    const int c = (int)(idx % L);
    const long t = idx / L;
    const int l = (int)(t % k);
    const int w = (int)(t / k);
    const double v = unp[(size_t)l * L + c];
    lo[((size_t)w * nu + nd + l) * L + c] = static_cast<float>(v - static_cast<double>(static_cast<float>(v)));
  }
}

cudaError_t launch_fill_unpaired_lo(const DevSystem &s, float *lo, int W, cudaStream_t st) {
  if (W <= 0 || s.n_up == s.n_dn) return cudaSuccess;
  const long total = (long)W * (s.n_up - s.n_dn) * s.L;
  long blocks = (total + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  k_fill_unpaired_lo<<<(int)blocks, 256, 0, st>>>(s.unpaired, lo, W, s.n_up, s.n_dn, s.L);
  return cudaGetLastError();
}
template cudaError_t launch_fill_unpaired<float>(const DevSystem &, float *, int, cudaStream_t);

// 1/p in FP64 from an FP32 seed and two Newton steps y <- y (2 - p y) (error
// squares each step: 2^-23 -> 2^-46 -> below FP64 rounding); p must be a
// normal number within FP32 range, else the FP64 division is used.
__device__ __forceinline__ double recip_newton(double p) {
  const double a = fabs(p);
  if (!(a > 1e-37 && a < 1e37)) return 1.0 / p;
  double y = static_cast<double>(__frcp_rn(static_cast<float>(p)));
  y = y * fma(-p, y, 2.0);
  y = y * fma(-p, y, 2.0);
  return y;
}

// x / p for the clustered elimination, where every CTA of the walker waits for the
// pivot row: three FP64 instructions (165 clocks each) from p to the result.  The
// FP32 seed y is taken and put back by integer instructions, e = 1 - p y, and
// x / p = x y (1 + e + e^2) up to e^3 < 2^-63.  1/p as above and a product take
// nine, conversions and range checks included (64 walkers of N_up = 256: 3.5 -> 3.2
// ms; no gain for N_up <= 64, whose CTAs hide it).
struct PivotRecip {
  double y, t;
  __device__ __forceinline__ explicit PivotRecip(double p) {
    const int hi = __double2hiint(p), lo = __double2loint(p);
    const int ef = ((hi >> 20) & 0x7ff) - 896;  // FP32's exponent field
    if (ef < 4 || ef > 250) {
      y = 1.0 / p;
      t = 0.0;
      return;
    }
    // p truncated to FP32, its reciprocal, and that as FP64
    const int r = __float_as_int(__frcp_rn(__int_as_float(
        (hi & 0x80000000) | (ef << 23) | ((hi & 0xfffff) << 3) | static_cast<int>(static_cast<unsigned>(lo) >> 29))));
    y = __hiloint2double((r & 0x80000000) | ((((r >> 23) & 0xff) + 896) << 20) | ((r & 0x7fffff) >> 3), r << 29);
    const double e = fma(-p, y, 1.0);
    t = fma(e, e, e);
  }
  __device__ __forceinline__ double value() const { return fma(y, t, y); }
  __device__ __forceinline__ double times(double x) const {
    const double q = x * y;
    return fma(q, t, q);
  }
};

// log|prod of pivots| without a logarithm per pivot: the product is kept as a
// mantissa in [1/2, 1) and a binary exponent (frexp after every factor), and
// one log at the end gives log|m| + E ln 2.
struct PivotProduct {
  double m = 1.0;
  int e = 0;
  __device__ __forceinline__ void mul(double pv) {
    int e1, e2;
    const double a = frexp(fabs(pv), &e1);
    m = frexp(m * a, &e2);
    e += e1 + e2;
  }
  __device__ __forceinline__ double log_abs() const { return log(m) + e * 0.6931471805599453; }
};

// ---------------------------------------------------------------------------
// FP64 refresh: Gauss-Jordan elimination with partial pivoting.  log|det G~| is
// log|prod of pivots|, the sign the product of pivot signs and the parity of
// the row order.  The fresh inverse replaces the Sherman-Morrison one; their
// largest difference times max|G~| is the walker's drift.
// ---------------------------------------------------------------------------
constexpr size_t kMmatSmemMax = 200 * 1024;  // k_mmat stages G~^{-1} whole up to this footprint
constexpr size_t kRefreshSmemMax = 200 * 1024;  // shared-memory rows of the in-place refresh up to this footprint

// N_up <= 32: register-resident in-place Gauss-Jordan.  A group of NM lanes
// (NM = 8, 16 or 32, the smallest >= N_up) holds one walker's matrix, lane c
// its column c in NM registers (rows and columns past N_up are the identity);
// a warp holds 32 / NM walkers.  No rows are swapped: step k pivots on the
// largest |entry| of column k among the rows not yet pivoted (the lowest row
// on ties), with the in-place update of the exchange form (pivot row scaled by
// 1/p, -f_i / p into column k, f_i = A[i][k]).  After the last step row p_k
// holds x_k, so inverse[k][p_k'] is entry (p_k, k') of the result, and the
// determinant's sign is that of the pivot product times (-1)^(inversions of
// the pivot order).  Pivot keys compare as the integer bits of |value|.
template <typename T, int NM>
struct RefreshInverseReg {
  static __device__ __forceinline__ void run(const double *__restrict__ gm, T *__restrict__ ginv,
                                             double *__restrict__ scal, int *__restrict__ status, int n, int W,
                                             int check_drift, double drift_tol, double *__restrict__ ginv64,
                                             const uint3 bid, const uint3 gdim) {
    assume_global(gm, ginv, scal, status);
    constexpr int kGroups = 32 / NM;
    constexpr unsigned kFull = 0xffffffffu;
    const int lane = threadIdx.x & 31, c = lane & (NM - 1), g0 = lane - c;
    const int w = (bid.x * 4 + (threadIdx.x >> 5)) * kGroups + lane / NM;
    const bool live = w < W;  // lanes of walkers past W run on the identity and write nothing
    const double *Gw = gm + (size_t)(live ? w : 0) * n * n;
    double a[NM];
    double gmax = 0.0;
  #pragma unroll
    for (int i = 0; i < NM; ++i) {
      double v = i == c ? 1.0 : 0.0;
      if (live && i < n && c < n) {
        v = Gw[i * n + c];
        gmax = fmax(gmax, fabs(v));
      }
      a[i] = v;
    }
    const unsigned rows_n = n >= 32 ? kFull : ((1u << n) - 1u);
    unsigned used = 0;  // rows pivoted so far (the same in every lane of a group)
    int inversions = 0, myp = 0, myq = 0;  // lane c: pivot row of step c; step at which row c was pivoted
    PivotProduct pp;
    bool neg = false, ok = true;
    for (int k = 0; k < n; ++k) {
      // lane i of the group picks up f_i = A[i][k] from lane k
      double fme = 0.0;
  #pragma unroll
      for (int i = 0; i < NM; ++i) {
        const double t = __shfl_sync(kFull, a[i], g0 + k);
        if (c == i) fme = t;
      }
      unsigned long long key = (c < n && !((used >> c) & 1u))
                                   ? static_cast<unsigned long long>(__double_as_longlong(fme)) & 0x7fffffffffffffffull
                                   : 0ull;
      int pi = c;
  #pragma unroll
      for (int o = NM / 2; o > 0; o >>= 1) {
        const unsigned long long ok2 = __shfl_xor_sync(kFull, key, o);
        const int oi = __shfl_xor_sync(kFull, pi, o);
        if (ok2 > key || (ok2 == key && oi < pi)) {
          key = ok2;
          pi = oi;
        }
      }
      const int p = pi;
      const double pv = __shfl_sync(kFull, fme, g0 + p);
      ok = ok && !((used >> p) & 1u) && pv != 0.0 && isfinite(pv);
      inversions += __popc(~used & rows_n & ((1u << p) - 1u));
      used |= 1u << p;
      if (c == k) myp = p;
      if (c == p) myq = k;
      pp.mul(pv);
      neg ^= pv < 0.0;
      const double ip = recip_newton(pv);
      double prow = 0.0;
  #pragma unroll
      for (int i = 0; i < NM; ++i)
        if (i == p) prow = a[i];
      prow = c == k ? ip : prow * ip;
      const bool colk = c == k;
  #pragma unroll
      for (int i = 0; i < NM; ++i) {
        const double fi = __shfl_sync(kFull, a[i], g0 + k);
        a[i] = i == p ? prow : fma(-fi, prow, colk ? 0.0 : a[i]);
      }
    }
    // inverse[k][p_c] = result[p_k][c]: row i of the result goes to row q_i
    T *gi = ginv + (size_t)(live ? w : 0) * n * n;
    double dmax = 0.0;
  #pragma unroll
    for (int i = 0; i < NM; ++i) {
      const int qi = __shfl_sync(kFull, myq, g0 + i);
      if (live && ok && i < n && c < n) {
        const size_t idx = (size_t)qi * n + myp;
        if (check_drift) dmax = fmax(dmax, fabs(a[i] - static_cast<double>(gi[idx])));
        gi[idx] = static_cast<T>(a[i]);
        if (ginv64) ginv64[(size_t)w * n * n + idx] = a[i];
      }
    }
  #pragma unroll
    for (int o = NM / 2; o > 0; o >>= 1) {
      dmax = fmax(dmax, __shfl_xor_sync(kFull, dmax, o));
      gmax = fmax(gmax, __shfl_xor_sync(kFull, gmax, o));
    }
    if (!live || c != 0) return;
    double *sw = scal + (size_t)w * S_STRIDE;
    if (!ok) {
      status[w] |= JAGP_WS_SINGULAR;
      sw[S_LOGDET] = -INFINITY;
      sw[S_SIGN] = 0.0;
      return;
    }
    sw[S_LOGDET] = pp.log_abs();
    sw[S_SIGN] = (neg != (inversions & 1)) ? -1.0 : 1.0;
    if (check_drift) {
      const double drift = dmax * gmax;
      sw[S_DRIFT] = drift;
      if (!(drift <= drift_tol)) status[w] |= JAGP_WS_DRIFT;
    }
}
};
template <typename T, int NM>
__global__ void __launch_bounds__(128) k_refresh_inverse_reg(const double *__restrict__ gm, T *__restrict__ ginv,
                                                             double *__restrict__ scal, int *__restrict__ status,
                                                             int n, int W, int check_drift, double drift_tol,
                                                             double *__restrict__ ginv64) {
  RefreshInverseReg<T, NM>::run(gm, ginv, scal, status, n, W, check_drift, drift_tol, ginv64, blockIdx, gridDim);
}

// The pivot of a step over a warp: the largest |f| of the rows that are still to
// be pivoted (key: the integer bits of |f|, 0 for the others), the lowest row on ties.
__device__ __forceinline__ int best_row(unsigned long long key, int row) {
  constexpr unsigned kFull = 0xffffffffu;
  const unsigned hi = static_cast<unsigned>(key >> 32), lo = static_cast<unsigned>(key);
  const unsigned mh = __reduce_max_sync(kFull, hi);
  const unsigned ml = __reduce_max_sync(kFull, hi == mh ? lo : 0u);
  return static_cast<int>(__reduce_min_sync(kFull, hi == mh && lo == ml ? static_cast<unsigned>(row) : 0xffffu));
}
__device__ __forceinline__ unsigned long long abs_key(double f) {
  return static_cast<unsigned long long>(__double_as_longlong(f)) & 0x7fffffffffffffffull;
}

// log|det| and the parity of negative pivots from two pivots per lane (1 where
// there is none): the mantissas multiplied and the exponents added over the
// warp, one log at the end
__device__ __forceinline__ double log_pivots(double first, double second, bool *neg) {
  int e1, e2;
  double m = frexp(fabs(first), &e1) * frexp(fabs(second), &e2);
  int e = e1 + e2;
  unsigned flips = (__double_as_longlong(first) < 0) ^ (__double_as_longlong(second) < 0);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m *= __shfl_xor_sync(0xffffffffu, m, o);  // at most 64 factors of at least 1/2
    e += __shfl_xor_sync(0xffffffffu, e, o);
    flips ^= __shfl_xor_sync(0xffffffffu, flips, o);
  }
  *neg = flips & 1u;
  return log(m) + e * 0.6931471805599453;
}

// 32 < N_up <= 16 CPL (CPL = 3 or 4): the same elimination on four warps of one
// walker per CTA.  Half-warp g = 0 .. 7 holds the rows g + 8 i, its lane c the
// columns c + 16 j (identity past N_up), so that the FP64 pipe, which bounds a
// step, sees little padding (at N_up = 44: 66 FMA warp instructions a step
// against 60.5 without any; two columns c, c + 32 per lane took 88).  Column k goes
// to shared memory, every warp finds the pivot, the pivot row's half-warp
// publishes it scaled, and all update.  Two barriers a step; the exchange
// slots alternate with the parity of k, so no third is needed.  Measured
// (serialised): 509 walkers of N_up = 44 342 -> 193 us against two warps per
// walker with two columns per lane and the multipliers through shuffles;
// the FP64 instructions alone take 110 us.
template <typename T, int CPL>
struct RefreshInverseCta {
  static constexpr int kMinBlocks = 4;
  static __device__ __forceinline__ void run(const double *__restrict__ gm, T *__restrict__ ginv,
                                             double *__restrict__ scal, int *__restrict__ status, int n, int W,
                                             int check_drift, double drift_tol, double *__restrict__ ginv64,
                                             const uint3 bid, const uint3 gdim) {
    assume_global(gm, ginv, scal, status);
    constexpr unsigned kFull = 0xffffffffu;
    constexpr int RPL = 2 * CPL;
    __shared__ double s_f[2][64], s_prow[2][64], s_pv[64];
    __shared__ int s_q[64], s_p[64];  // step at which each row was pivoted; pivot row of each step
    __shared__ double s_red[4][2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = lane & 15, g = 2 * warp + (lane >> 4);
    const int w = bid.x;
    const double *Gw = gm + (size_t)w * n * n;
    double a[RPL][CPL];
    double gmax = 0.0;
  #pragma unroll
    for (int i = 0; i < RPL; ++i)
  #pragma unroll
      for (int j = 0; j < CPL; ++j) {
        const int r = g + 8 * i, col = c + 16 * j;
        double v = r == col ? 1.0 : 0.0;
        if (r < n && col < n) {
          v = Gw[(size_t)r * n + col];
          gmax = fmax(gmax, fabs(v));
        }
        a[i][j] = v;
      }
    unsigned long long used = 0;
    const unsigned long long rows_n = n >= 64 ? ~0ull : ((1ull << n) - 1ull);
    int inversions = 0;
    bool ok = true;
  #pragma unroll
    for (int jj = 0; jj < CPL; ++jj) {
      for (int kk = 0; kk < 16; ++kk) {
        const int k = 16 * jj + kk, par = k & 1;
        if (k >= n) break;
        if (c == kk) {
  #pragma unroll
          for (int i = 0; i < RPL; ++i) s_f[par][g + 8 * i] = a[i][jj];
        }
        __syncthreads();
        // rows lane and lane + 32: the better of the two, then over the warp
        const double f0 = s_f[par][lane], f1 = s_f[par][lane + 32];
        const unsigned long long k0 = !((used >> lane) & 1ull) ? abs_key(f0) : 0ull;
        const unsigned long long k1 = lane + 32 < n && !((used >> (lane + 32)) & 1ull) ? abs_key(f1) : 0ull;
        const int p = best_row(k1 > k0 ? k1 : k0, k1 > k0 ? lane + 32 : lane);
        const double pv = s_f[par][p];
        const unsigned long long pk = abs_key(pv);
        ok = ok && !((used >> p) & 1ull) && pk != 0ull && pk < 0x7ff0000000000000ull;
        inversions += __popcll(~used & rows_n & ((1ull << p) - 1ull));
        used |= 1ull << p;
        if (threadIdx.x == 0) {
          s_q[p] = k;
          s_p[k] = p;
          s_pv[k] = pv;
        }
        if (warp == (p & 7) >> 1) {  // the warp with the pivot row (lane half (p & 7) & 1) publishes it scaled
          const double ip = recip_newton(pv);
          double x[CPL];
  #pragma unroll
          for (int j = 0; j < CPL; ++j) x[j] = a[0][j];
  #pragma unroll
          for (int i = 1; i < RPL; ++i)
            if (i == p >> 3) {
  #pragma unroll
              for (int j = 0; j < CPL; ++j) x[j] = a[i][j];
            }
          if (g == (p & 7)) {
  #pragma unroll
            for (int j = 0; j < CPL; ++j) s_prow[par][c + 16 * j] = j == jj && c == kk ? ip : x[j] * ip;
          }
        }
        __syncthreads();
        double v[CPL];
  #pragma unroll
        for (int j = 0; j < CPL; ++j) v[j] = s_prow[par][c + 16 * j];
  #pragma unroll
        for (int i = 0; i < RPL; ++i) {
          if (2 * warp + 8 * i < n) {  // warp-uniform: at least one of the two halves' rows exists
            const int r = g + 8 * i;
            const double f = s_f[par][r];
  #pragma unroll
            for (int j = 0; j < CPL; ++j) {
              const double base = j == jj && c == kk ? 0.0 : a[i][j];
              a[i][j] = r == p ? v[j] : fma(-f, v[j], base);
            }
          }
        }
      }
    }
    __syncthreads();  // s_q, s_p, s_pv complete
    // inverse[k][p_c] = result[p_k][c]: row r of the result goes to row q_r, column c to column p_c
    T *gi = ginv + (size_t)w * n * n;
    double dmax = 0.0;
    if (ok) {
  #pragma unroll
      for (int i = 0; i < RPL; ++i) {
        const int r = g + 8 * i;
        if (r >= n) continue;
        const size_t row = (size_t)s_q[r] * n;
  #pragma unroll
        for (int j = 0; j < CPL; ++j) {
          const int col = c + 16 * j;
          if (col >= n) continue;
          const size_t idx = row + s_p[col];
          if (check_drift) dmax = fmax(dmax, fabs(a[i][j] - static_cast<double>(gi[idx])));
          gi[idx] = static_cast<T>(a[i][j]);
          if (ginv64) ginv64[(size_t)w * n * n + idx] = a[i][j];
        }
      }
    }
  #pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      dmax = fmax(dmax, __shfl_xor_sync(kFull, dmax, o));
      gmax = fmax(gmax, __shfl_xor_sync(kFull, gmax, o));
    }
    if (lane == 0) {
      s_red[warp][0] = gmax;
      s_red[warp][1] = dmax;
    }
    __syncthreads();
    if (warp != 0) return;
    bool neg;
    const double logdet = log_pivots(ok ? s_pv[lane] : 1.0, ok && lane + 32 < n ? s_pv[lane + 32] : 1.0, &neg);
    if (lane != 0) return;
    double *sw = scal + (size_t)w * S_STRIDE;
    if (!ok) {
      status[w] |= JAGP_WS_SINGULAR;
      sw[S_LOGDET] = -INFINITY;
      sw[S_SIGN] = 0.0;
      return;
    }
    sw[S_LOGDET] = logdet;
    sw[S_SIGN] = (neg != ((inversions & 1) != 0)) ? -1.0 : 1.0;
    if (check_drift) {
      const double gm4 = fmax(fmax(s_red[0][0], s_red[1][0]), fmax(s_red[2][0], s_red[3][0]));
      const double dm4 = fmax(fmax(s_red[0][1], s_red[1][1]), fmax(s_red[2][1], s_red[3][1]));
      const double drift = dm4 * gm4;
      sw[S_DRIFT] = drift;
      if (!(drift <= drift_tol)) status[w] |= JAGP_WS_DRIFT;
    }
}
};
template <typename T, int CPL>
__global__ void __launch_bounds__(128, 4) k_refresh_inverse_cta(const double *__restrict__ gm, T *__restrict__ ginv,
                                                                double *__restrict__ scal, int *__restrict__ status,
                                                                int n, int W, int check_drift, double drift_tol,
                                                                double *__restrict__ ginv64) {
  RefreshInverseCta<T, CPL>::run(gm, ginv, scal, status, n, W, check_drift, drift_tol, ginv64, blockIdx, gridDim);
}

// N_up > 64 while a cluster's shared memory holds the matrix: the same elimination
// (no row swaps) on a cluster of cl CTAs per walker, CTA c with the columns c C ..
// c C + C - 1 of every row in shared memory.  The owner of column k finds the
// pivot row and sends the column and the row's index to every CTA; the rest of a
// step is local (each CTA has its columns of the pivot row), so a step costs one
// cluster barrier, and the column buffers alternate with the parity of k.  A
// thread keeps one column and takes every R-th row, R = threads / C, so that
// consecutive threads touch consecutive elements and none of the FP64 pipe, which
// bounds an update (n C / 2 clocks), goes to padding.  64 walkers of N_up = 256: 6.4 ms
// in place in global memory, 3.2 so.  Several CTAs share an SM and
// hide each other's barriers and pivot searches.
constexpr int kClusterThreads = 256;
struct ClusterSmem {
  static __host__ __device__ size_t bytes(int n, int C) {
    // the columns, two column buffers, the scaled pivot row, pivots; pivot rows, steps, used flags
    return ((size_t)n * C + 3 * (size_t)n + C) * sizeof(double) + (size_t)3 * n * sizeof(int);
  }
};

template <typename T>
struct RefreshInverseCluster {
  static __device__ __forceinline__ void run(const double *__restrict__ gm, T *__restrict__ ginv,
                                             double *__restrict__ scal, int *__restrict__ status, int n, int cl,
                                             int check_drift, double drift_tol, double *__restrict__ ginv64,
                                             const uint3 bid, const uint3 gdim) {
    assume_global(gm, ginv, scal, status);
    namespace cg = cooperative_groups;
    extern __shared__ double sm[];
    const int C = (n + cl - 1) / cl, w = (int)bid.x / cl, rank = (int)bid.x - w * cl;
    double *const S = sm;                      // [n][C]
    double *const F = S + (size_t)n * C;       // [2][n] column k before the step
    double *const prow = F + 2 * n;            // [C]
    double *const pvs = prow + C;              // [n] pivots
    int *const sp = reinterpret_cast<int *>(pvs + n);  // [n] pivot row of each step
    int *const sq = sp + n;                    // [n] step at which each row was pivoted
    int *const used = sq + n;                  // [n]
    __shared__ int s_piv[2];
    __shared__ double red[kClusterThreads / 32][2];
    __shared__ double s_max[8][2];             // rank 0: every CTA's largest |G~| and drift
    __shared__ unsigned s_par[kClusterThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto cluster_sync = [&] {
      if (cl > 1) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
      } else {
        __syncthreads();
      }
    };
    // the CTA's copy of p in rank r's shared memory
    auto remote = [&](auto *q, int r) { return cl > 1 ? cg::this_cluster().map_shared_rank(q, r) : q; };
    const int j0 = rank * C, nc = n - j0 < C ? (n - j0 > 0 ? n - j0 : 0) : C;  // this CTA's columns
    const int R = kClusterThreads / C, g = tid / C, jc = tid - g * C;  // (C <= kClusterThreads)
    const double *Gw = gm + (size_t)w * n * n;
    double gmax = 0.0;
    for (int i = warp; i < n; i += kClusterThreads / 32)
      for (int j = lane; j < C; j += 32) {
        const double v = j < nc ? Gw[(size_t)i * n + j0 + j] : 0.0;
        gmax = fmax(gmax, fabs(v));
        S[(size_t)i * C + j] = v;
      }
    for (int i = tid; i < n; i += kClusterThreads) used[i] = 0;
    bool ok = true;
    cluster_sync();  // (every CTA of the cluster runs, its buffers may be written)
    for (int k = 0; k < n; ++k) {
      const int par = k & 1, owner = k / C, kc = k - owner * C;
      double *const f = F + par * n;
      if (rank == owner) {
        // column k to every CTA; the pivot among the rows not yet used
        for (int i = tid; i < n; i += kClusterThreads) {
          const double v = S[(size_t)i * C + kc];
          for (int r = 0; r < cl; ++r) remote(f, r)[i] = v;
        }
        if (warp == 0) {
          unsigned long long key = 0ull;
          int row = lane;
#pragma unroll 4
          for (int i = lane; i < n; i += 32) {
            const unsigned long long ki = used[i] ? 0ull : abs_key(S[(size_t)i * C + kc]);
            if (ki > key) {
              key = ki;
              row = i;
            }
          }
          const int p = best_row(key, row);
          if (lane < cl) *remote(&s_piv[par], lane) = p;
        }
      }
      cluster_sync();
      const int p = s_piv[par];
      const double pv = f[p];
      const unsigned long long pk = abs_key(pv);
      if (used[p] || pk == 0ull || pk >= 0x7ff0000000000000ull) {  // the same in every CTA
        ok = false;
        break;
      }
      const bool mine = rank == owner;
      // (the reciprocal only where a warp has elements of the pivot row: it costs as
      // much of the FP64 pipe as a third of an update when every warp forms it)
      if (tid < C) {  // (C <= kClusterThreads)
        const PivotRecip ip(pv);
        prow[tid] = mine && tid == kc ? ip.value() : ip.times(S[(size_t)p * C + tid]);
      }
      __syncthreads();
      if (tid == 0) {
        sp[k] = p;
        sq[p] = k;
        pvs[k] = pv;
        used[p] = 1;
      }
      if (g < R) {
        const double x = prow[jc];
        const bool ck = mine && jc == kc;
        double *Sj = S + jc;
#pragma unroll 8
        for (int i = g; i < n; i += R) {
          const double base = ck ? 0.0 : Sj[i * C];
          Sj[i * C] = i == p ? x : fma(-f[i], x, base);
        }
      }
      __syncthreads();
    }
    T *gi = ginv + (size_t)w * n * n;
    double dmax = 0.0;
    if (ok) {
      // inverse[k][p_c] = result[p_k][c]: row i of the result goes to row q_i, column c to column p_c
      for (int i = warp; i < n; i += kClusterThreads / 32) {
        const size_t row = (size_t)sq[i] * n;
        for (int j = lane; j < nc; j += 32) {
          const double v = S[(size_t)i * C + j];
          const size_t idx = row + sp[j0 + j];
          if (check_drift) dmax = fmax(dmax, fabs(v - static_cast<double>(gi[idx])));
          gi[idx] = static_cast<T>(v);
          if (ginv64) ginv64[(size_t)w * n * n + idx] = v;
        }
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
      gmax = fmax(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
    }
    if (lane == 0) {
      red[warp][0] = gmax;
      red[warp][1] = dmax;
    }
    // parity of the pivot order
    unsigned inv = 0;
    if (ok && rank == 0)
      for (int k = tid; k < n; k += kClusterThreads)
        for (int q = k + 1; q < n; ++q) inv ^= sp[q] < sp[k];
    inv = __reduce_xor_sync(0xffffffffu, inv);
    if (lane == 0) s_par[warp] = inv;
    __syncthreads();
    if (tid == 0) {
      for (int q = 1; q < kClusterThreads / 32; ++q) {
        gmax = fmax(gmax, red[q][0]);
        dmax = fmax(dmax, red[q][1]);
      }
      double *m = remote(&s_max[0][0], 0);
      m[2 * rank] = gmax;
      m[2 * rank + 1] = dmax;
    }
    cluster_sync();
    if (rank != 0 || warp != 0) return;
    double *sw = scal + (size_t)w * S_STRIDE;
    if (!ok) {
      if (lane == 0) {
        status[w] |= JAGP_WS_SINGULAR;
        sw[S_LOGDET] = -INFINITY;
        sw[S_SIGN] = 0.0;
      }
      return;
    }
    // log|det|: each lane's pivots as a mantissa and an exponent, then the warp's
    PivotProduct pp;
    unsigned flips = 0;
    for (int k = lane; k < n; k += 32) {
      pp.mul(pvs[k]);
      flips ^= pvs[k] < 0.0;
    }
    double mant = pp.m;
    int e = pp.e;
    for (int o = 16; o > 0; o >>= 1) {
      mant *= __shfl_xor_sync(0xffffffffu, mant, o);
      e += __shfl_xor_sync(0xffffffffu, e, o);
    }
    flips = __reduce_xor_sync(0xffffffffu, flips);
    if (lane != 0) return;
    for (int q = 0; q < kClusterThreads / 32; ++q) flips ^= s_par[q];
    sw[S_LOGDET] = log(mant) + e * 0.6931471805599453;
    sw[S_SIGN] = flips ? -1.0 : 1.0;
    if (check_drift) {
      double g = 0.0, d = 0.0;
      for (int r = 0; r < cl; ++r) {
        g = fmax(g, s_max[r][0]);
        d = fmax(d, s_max[r][1]);
      }
      const double drift = d * g;
      sw[S_DRIFT] = drift;
      if (!(drift <= drift_tol)) status[w] |= JAGP_WS_DRIFT;
    }
}
};
template <typename T>
__global__ void __launch_bounds__(kClusterThreads) k_refresh_inverse_cluster(
    const double *__restrict__ gm, T *__restrict__ ginv, double *__restrict__ scal, int *__restrict__ status, int n,
    int cl, int check_drift, double drift_tol, double *__restrict__ ginv64) {
  RefreshInverseCluster<T>::run(gm, ginv, scal, status, n, cl, check_drift, drift_tol, ginv64, blockIdx, gridDim);
}

// In-place Gauss-Jordan (larger N_up): step k scales the pivot row, stores
// -f_i / p in column k and updates the rest, so the inverse takes the place of
// G~ (half the work of eliminating [G~ | I]); the row swaps of the partial
// pivoting become column swaps of the result, undone in reverse order at the
// end.  Rows i < rs are copied to shared memory (row pitch n + 1); the others
// are overwritten in global memory, where they stay L2-resident while the CTA
// works on them (the launch keeps one CTA per SM, so the resident rows of all
// CTAs together fit in L2).
template <typename T>
struct RefreshInverseInplace {
  static __device__ __forceinline__ void run(double *__restrict__ gm, T *__restrict__ ginv, double *__restrict__ scal,
                                             int *__restrict__ status, int n, int rs, int check_drift,
                                             double drift_tol, double *__restrict__ ginv64, const uint3 bid,
                                             const uint3 gdim) {
    assume_global(gm, ginv, scal, status);
    extern __shared__ double sm[];
    const int ld = n + 1;
    double *prow = sm + (size_t)rs * ld;          // n: the scaled pivot row
    double *f = prow + n;                         // n: column k before the step
    int *perm = reinterpret_cast<int *>(f + n);   // n: pivot row of each step
    __shared__ int s_piv;
    __shared__ double s_pv;
    __shared__ double red[32];
    const int tid = threadIdx.x, bs = blockDim.x, w = bid.x, lane = tid & 31, warp = tid >> 5, nw = bs >> 5;
    double *const G = gm + (size_t)w * n * n;
    auto R = [&](int i) -> double * { return i < rs ? sm + (size_t)i * ld : G + (size_t)i * n; };
    double gmax = 0.0;
    for (int idx = tid; idx < n * n; idx += bs) {
      const int i = idx / n, j = idx - i * n;
      const double v = G[idx];
      gmax = fmax(gmax, fabs(v));
      if (i < rs) sm[(size_t)i * ld + j] = v;
    }
    PivotProduct pp;
    double sgn = 1.0;
    bool ok = true;
    __syncthreads();
    for (int k = 0; k < n; ++k) {
      if (warp == 0) {
        double best = -1.0;
        int bi = k;
        for (int i = k + lane; i < n; i += 32) {
          const double v = fabs(R(i)[k]);
          if (v > best) {
            best = v;
            bi = i;
          }
        }
  #pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const double ob = __shfl_xor_sync(0xffffffffu, best, o);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
          if (ob > best || (ob == best && oi < bi)) {
            best = ob;
            bi = oi;
          }
        }
        if (lane == 0) {
          s_piv = bi;
          s_pv = R(bi)[k];
        }
      }
      __syncthreads();
      const int p = s_piv;
      const double pv = s_pv;
      if (!(pv != 0.0) || !isfinite(pv)) {
        ok = false;
        break;
      }
      if (p != k) {
        double *Rk = R(k), *Rp = R(p);
        for (int j = tid; j < n; j += bs) {
          const double t = Rk[j];
          Rk[j] = Rp[j];
          Rp[j] = t;
        }
        sgn = -sgn;
      }
      pp.mul(pv);
      if (pv < 0.0) sgn = -sgn;
      if (tid == 0) perm[k] = p;
      __syncthreads();
      const double ip = recip_newton(pv);
      {
        const double *Rk = R(k);
        for (int j = tid; j < n; j += bs) prow[j] = j == k ? ip : Rk[j] * ip;
      }
      for (int i = tid; i < n; i += bs) f[i] = i == k ? 0.0 : R(i)[k];
      __syncthreads();
      for (int i = warp; i < n; i += nw) {
        double *Ai = R(i);
        if (i == k) {
          for (int j = lane; j < n; j += 32) Ai[j] = prow[j];
        } else {
          // eight columns per lane at a time, all loads before the stores, so
          // that they are in flight together (Ai may be global memory)
          const double fi = f[i];
          for (int jb = 0; jb < n; jb += 256) {
            double v[8];
  #pragma unroll
            for (int t = 0; t < 8; ++t) {
              const int j = jb + lane + 32 * t;
              v[t] = j < n ? Ai[j] : 0.0;
            }
  #pragma unroll
            for (int t = 0; t < 8; ++t) {
              const int j = jb + lane + 32 * t;
              if (j < n) Ai[j] = fma(-fi, prow[j], v[t]);
            }
          }
        }
      }
      __syncthreads();
      // column k of the other rows: -f_i / p (replacing what the update left there)
      for (int i = tid; i < n; i += bs)
        if (i != k) R(i)[k] = -f[i] * ip;
      __syncthreads();
    }
    T *gi = ginv + (size_t)w * n * n;
    if (!ok) {
      if (tid == 0) {
        status[w] |= JAGP_WS_SINGULAR;
        scal[(size_t)w * S_STRIDE + S_LOGDET] = -INFINITY;
        scal[(size_t)w * S_STRIDE + S_SIGN] = 0.0;
      }
      return;
    }
    for (int k = n - 1; k >= 0; --k) {
      const int p = perm[k];
      if (p != k)
        for (int i = tid; i < n; i += bs) {
          double *Ai = R(i);
          const double t = Ai[k];
          Ai[k] = Ai[p];
          Ai[p] = t;
        }
      __syncthreads();
    }
    double dmax = 0.0;
    for (int idx = tid; idx < n * n; idx += bs) {
      const double v = R(idx / n)[idx % n];
      if (check_drift) dmax = fmax(dmax, fabs(v - static_cast<double>(gi[idx])));
      gi[idx] = static_cast<T>(v);
      if (ginv64) ginv64[(size_t)w * n * n + idx] = v;
    }
    for (int o = 16; o > 0; o >>= 1) {
      dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
      gmax = fmax(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
    }
    if (lane == 0) {
      red[warp] = dmax;
      red[16 + warp] = gmax;
    }
    __syncthreads();
    if (tid == 0) {
      double d = 0.0, g = 0.0;
      for (int q = 0; q < nw; ++q) {
        d = fmax(d, red[q]);
        g = fmax(g, red[16 + q]);
      }
      scal[(size_t)w * S_STRIDE + S_LOGDET] = pp.log_abs();
      scal[(size_t)w * S_STRIDE + S_SIGN] = sgn;
      if (check_drift) {
        const double drift = d * g;
        scal[(size_t)w * S_STRIDE + S_DRIFT] = drift;
        if (!(drift <= drift_tol)) status[w] |= JAGP_WS_DRIFT;
      }
    }
}
};
template <typename T>
__global__ void __launch_bounds__(512) k_refresh_inverse_inplace(double *__restrict__ gm, T *__restrict__ ginv,
                                                                 double *__restrict__ scal, int *__restrict__ status,
                                                                 int n, int rs, int check_drift, double drift_tol,
                                                                 double *__restrict__ ginv64) {
  RefreshInverseInplace<T>::run(gm, ginv, scal, status, n, rs, check_drift, drift_tol, ginv64, blockIdx, gridDim);
}


template <typename T>
cudaError_t launch_refresh_inverse(double *gm, T *ginv, double *scal, int *status, int n, int W,
                                   int check_drift, double drift_tol, cudaStream_t st, double *ginv64) {
  if (W <= 0) return cudaSuccess;
  if (n > 32 && n <= 48 && !group_recorder())  // (grouped launches: one kernel for both sizes)
    return launch_or_record<RefreshInverseCta<T, 3>, 128>(k_refresh_inverse_cta<T, 3>, dim3(W), dim3(128), 0, st, gm,
                                                          ginv, scal, status, n, W, check_drift, drift_tol, ginv64);
  if (n > 32 && n <= 64)
    return launch_or_record<RefreshInverseCta<T, 4>, 128>(k_refresh_inverse_cta<T, 4>, dim3(W), dim3(128), 0, st, gm,
                                                          ginv, scal, status, n, W, check_drift, drift_tol, ginv64);
  // a cluster per walker whose CTAs together hold the matrix: as few CTAs as fit, or
  // more (up to eight) while that leaves SMs idle or keeps a second CTA off an SM
  // (grouped launches: one CTA, up to N_up = 156)
  if (n > 64) {
    int cl = 1;
    auto fits = [&](int c, size_t limit) {
      return (n + c - 1) / c <= kClusterThreads && ClusterSmem::bytes(n, (n + c - 1) / c) <= limit;
    };
    const int most = group_recorder() ? 1 : 8;
    while (cl < most && (!fits(cl, kRefreshSmemMax) || (long long)W * cl < 2 * 152 || !fits(cl, kRefreshSmemMax / 2)))
      cl *= 2;
    if (fits(cl, kRefreshSmemMax)) {
      const size_t smem = ClusterSmem::bytes(n, (n + cl - 1) / cl);
      if (cl == 1)
        return launch_or_record<RefreshInverseCluster<T>, kClusterThreads>(
            k_refresh_inverse_cluster<T>, dim3(W), dim3(kClusterThreads), smem, st, (const double *)gm, ginv, scal,
            status, n, 1, check_drift, drift_tol, ginv64);
      static std::atomic<unsigned char> raised[64];
      cudaError_t e = group_raise_smem(reinterpret_cast<const void *>(k_refresh_inverse_cluster<T>), raised);
      if (e != cudaSuccess) return e;
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = static_cast<unsigned>(cl);
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      cfg.gridDim = dim3(W * cl);
      cfg.blockDim = dim3(kClusterThreads);
      cfg.dynamicSmemBytes = smem;
      cfg.stream = st;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      return cudaLaunchKernelEx(&cfg, k_refresh_inverse_cluster<T>, (const double *)gm, ginv, scal, status, n, cl,
                                check_drift, drift_tol, ginv64);
    }
    // as many leading rows in shared memory as fit in kRefreshSmemMax (which
    // also keeps one CTA per SM), the rest in global memory
    const size_t aux = (size_t)n * (2 * sizeof(double) + sizeof(int));
    const int rs = std::min(n, static_cast<int>((kRefreshSmemMax - aux) / ((size_t)(n + 1) * sizeof(double))));
    const size_t smem = (size_t)rs * (n + 1) * sizeof(double) + aux;
    return launch_or_record<RefreshInverseInplace<T>, 512>(k_refresh_inverse_inplace<T>, dim3(W), dim3(512), smem, st,
                                                           gm, ginv, scal, status, n, rs, check_drift, drift_tol,
                                                           ginv64);
  }
  if (n <= 32) {
    // 4 warps per CTA, 32 / NM walkers per warp
    if (n <= 8)
      return launch_or_record<RefreshInverseReg<T, 8>, 128>(k_refresh_inverse_reg<T, 8>, dim3((W + 15) / 16),
                                                            dim3(128), 0, st, gm, ginv, scal, status, n, W,
                                                            check_drift, drift_tol, ginv64);
    if (n <= 16)
      return launch_or_record<RefreshInverseReg<T, 16>, 128>(k_refresh_inverse_reg<T, 16>, dim3((W + 7) / 8),
                                                             dim3(128), 0, st, gm, ginv, scal, status, n, W,
                                                             check_drift, drift_tol, ginv64);
    return launch_or_record<RefreshInverseReg<T, 32>, 128>(k_refresh_inverse_reg<T, 32>, dim3((W + 3) / 4), dim3(128),
                                                           0, st, gm, ginv, scal, status, n, W, check_drift,
                                                           drift_tol, ginv64);
  }
  return cudaErrorInvalidValue;
}
template cudaError_t launch_refresh_inverse<double>(double *, double *, double *, int *, int, int, int, double,
                                                    cudaStream_t, double *);
template cudaError_t launch_refresh_inverse<float>(double *, float *, double *, int *, int, int, int, double,
                                                   cudaStream_t, double *);

// ---------------------------------------------------------------------------
// Kinetic-energy contraction vectors.  D = det G~ is linear in row i (up
// electron i) and in column j (down electron j), so
//   grad_i D / D = sum_mu grad phi_mu(r_i) M[i][mu],
//   up:   M[i]       = sum_j Ginv[j][i] Bt[j]      (Bt[j] = lambda phi(r_j^dn) or c^{(l)})
//   down: M[n_up + j] = sum_i Ginv[j][i] A_up[i]   (A_up[i] = phi(r_i^up)^T lambda)
// and the same M with the Laplacians.  One CTA per (walker, 64 columns).
// ---------------------------------------------------------------------------
struct Mmat {
  static __device__ __forceinline__ void run(DevSystem s, const double *__restrict__ ginv, const double *__restrict__ bt,
                                             const double *__restrict__ a_up, double *__restrict__ mbuf, const uint3 bid,
                                             const uint3 gdim) {
    assume_global(ginv, bt, a_up, mbuf);
    extern __shared__ double sm[];
    const int n = s.n_up, nd = s.n_dn, N = s.N, L = s.L;
    const int w = bid.y, c0 = bid.x * 64, tid = threadIdx.x;
    double *Gs = sm;              // n*n
    double *Bs = Gs + n * n;      // n*64
    double *As = Bs + n * 64;     // n*64
    for (int t = tid; t < n * n; t += 256) Gs[t] = ginv[(size_t)w * n * n + t];
    for (int t = tid; t < n * 64; t += 256) {
      const int j = t >> 6, c = t & 63;
      const bool in = c0 + c < L;
      Bs[t] = in ? bt[((size_t)w * n + j) * L + c0 + c] : 0.0;
      As[t] = in ? a_up[((size_t)w * n + j) * L + c0 + c] : 0.0;
    }
    __syncthreads();
    for (int idx = tid; idx < N * 64; idx += 256) {
      const int e = idx >> 6, c = idx & 63;
      if (c0 + c >= L) continue;
      double acc = 0.0;
      if (e < n) {
        for (int j = 0; j < n; ++j) acc = fma(Gs[j * n + e], Bs[j * 64 + c], acc);
      } else {
        const int jj = e - n;
        for (int i = 0; i < n; ++i) acc = fma(Gs[jj * n + i], As[i * 64 + c], acc);
      }
      (void)nd;
      mbuf[((size_t)w * N + e) * L + c0 + c] = acc;
    }
}
};
__global__ void __launch_bounds__(256) k_mmat(DevSystem s, const double *__restrict__ ginv, const double *__restrict__ bt,
                                              const double *__restrict__ a_up, double *__restrict__ mbuf) {
  Mmat::run(s, ginv, bt, a_up, mbuf, blockIdx, gridDim);
}

// The same contraction for N_up too large to stage G~^{-1} whole: 64 x 64
// output tiles (electrons x basis functions), 4 x 4 per thread, the sum over
// j (or i) in chunks of 16 in the same order as above.  Up tiles come first in
// blockIdx.y, then down tiles, so that no tile mixes the two formulas.
struct MmatTiled {
  static __device__ __forceinline__ void run(DevSystem s, const double *__restrict__ ginv, const double *__restrict__ bt,
                                             const double *__restrict__ a_up, double *__restrict__ mbuf, const uint3 bid,
                                             const uint3 gdim) {
    assume_global(ginv, bt, a_up, mbuf);
    __shared__ double Xs[16][64];  // Xs[k][e]: G~^{-1}[k][e] (up) or G~^{-1}[e][k] (down)
    __shared__ double Ys[16][64];  // Ys[k][c]: Bt[k][c] (up) or A_up[k][c] (down)
    const int n = s.n_up, N = s.N, L = s.L;
    const int w = bid.z, c0 = bid.x * 64, tid = threadIdx.x;
    const int up_tiles = (n + 63) / 64;
    const bool up = (int)bid.y < up_tiles;
    const int e0 = up ? bid.y * 64 : (bid.y - up_tiles) * 64;  // within the species
    const int ne = up ? n : s.n_dn;
    const double *G = ginv + (size_t)w * n * n;
    const double *Y = (up ? bt : a_up) + (size_t)w * n * L;
    const int tx = tid & 15, ty = tid >> 4;
    double acc[4][4];
  #pragma unroll
    for (int a = 0; a < 4; ++a)
  #pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
    for (int k0 = 0; k0 < n; k0 += 16) {
  #pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int idx = tid + q * 256;
        const int kk = idx >> 6, col = idx & 63, k = k0 + kk;
        double xv = 0.0, yv = 0.0;
        if (k < n) {
          const int e = e0 + col;
          if (e < ne) xv = up ? G[(size_t)k * n + e] : G[(size_t)e * n + k];
          if (c0 + col < L) yv = Y[(size_t)k * L + c0 + col];
        }
        Xs[kk][col] = xv;
        Ys[kk][col] = yv;
      }
      __syncthreads();
  #pragma unroll
      for (int kk = 0; kk < 16; ++kk) {
        double xa[4], yb[4];
  #pragma unroll
        for (int a = 0; a < 4; ++a) xa[a] = Xs[kk][ty * 4 + a];
  #pragma unroll
        for (int b = 0; b < 4; ++b) yb[b] = Ys[kk][tx * 4 + b];
  #pragma unroll
        for (int a = 0; a < 4; ++a)
  #pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] = fma(xa[a], yb[b], acc[a][b]);
      }
      __syncthreads();
    }
    const int ebase = up ? 0 : n;
  #pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int e = e0 + ty * 4 + a;
      if (e >= ne) continue;
      double *o = mbuf + ((size_t)w * N + ebase + e) * L;
  #pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int c = c0 + tx * 4 + b;
        if (c < L) o[c] = acc[a][b];
      }
    }
}
};
__global__ void __launch_bounds__(256) k_mmat_tiled(DevSystem s, const double *__restrict__ ginv, const double *__restrict__ bt,
                                                    const double *__restrict__ a_up, double *__restrict__ mbuf) {
  MmatTiled::run(s, ginv, bt, a_up, mbuf, blockIdx, gridDim);
}

// The mixed path's M vectors for small N_up on the CUDA cores: the sums of
// k_mmat with the FP64 inverse of the last refresh (split into two floats)
// against the two-float tables, as compensated dot products (error-free
// products and sums, the errors summed apart; Ogita, Rump and Oishi 2005) with
// the cross terms of the low parts, so that M + M_lo keeps about twice the
// FP32 precision.  One CTA per (walker, 64 columns); a thread takes a column and
// four electrons of one spin at a time, so that a table element serves four
// sums and the inverse comes as two 16-byte broadcasts per term: bound by the
// 13 FP32 instructions of a term (one output per thread read four operands
// from shared memory for each).  4096 walkers, N_up = 16, L = 320: 654 us with
// one output per thread.
constexpr int kMmatE = 4;

struct MmatDw {
  static __device__ __forceinline__ void run(DevSystem s, const double *__restrict__ ginv64,
                                             const float *__restrict__ bt, const float *__restrict__ bt_lo,
                                             const float *__restrict__ a_up, const float *__restrict__ a_lo,
                                             float *__restrict__ mbuf, float *__restrict__ mlo, const uint3 bid,
                                             const uint3 gdim) {
    assume_global(ginv64, bt, bt_lo, a_up, a_lo, mbuf, mlo);
    extern __shared__ float4 smf4[];
    const int n = s.n_up, nd = s.n_dn, N = s.N, L = s.L, ng = (n + kMmatE - 1) / kMmatE, np = ng * kMmatE;
    const int w = bid.y, c0 = bid.x * 64, tid = threadIdx.x;
    // per species, term j and electron e: (hi, lo) of Ginv[j][e] (up) or Ginv[e][j] (down), padded to np
    float2 *G = reinterpret_cast<float2 *>(smf4);            // [2][n][np]
    float2 *T = G + 2 * n * np;                                // [2][n][64]: Bt, A_up
    for (int t = tid; t < n * np; t += 256) {
      const int j = t / np, e = t - j * np;
      const fdw u = dw_of(e < n ? ginv64[(size_t)w * n * n + j * n + e] : 0.0);
      G[t] = make_float2(u.hi, u.lo);
    }
    for (int t = tid; t < n * np; t += 256) {
      const int e = t / n, j = t - e * n;  // (consecutive threads read a row of the inverse)
      const fdw d = dw_of(e < nd ? ginv64[(size_t)w * n * n + e * n + j] : 0.0);
      G[n * np + j * np + e] = make_float2(d.hi, d.lo);
    }
    for (int t = tid; t < n * 64; t += 256) {
      const int j = t >> 6, c = t & 63;
      const bool in = c0 + c < L;
      const size_t src = ((size_t)w * n + j) * L + c0 + c;
      T[t] = in ? make_float2(bt[src], bt_lo[src]) : make_float2(0.0f, 0.0f);
      T[n * 64 + t] = in ? make_float2(a_up[src], a_lo[src]) : make_float2(0.0f, 0.0f);
    }
    __syncthreads();
    const int c = tid & 63, groups = ng + (nd + kMmatE - 1) / kMmatE;
    if (c0 + c >= L) return;
    for (int g = tid >> 6; g < groups; g += 4) {
      const bool up = g < ng;
      const int e0 = (up ? g : g - ng) * kMmatE;
      const float2 *Gs = G + (up ? 0 : n * np) + e0, *Ts = T + (up ? 0 : n * 64) + c;
      float sh[kMmatE], err[kMmatE];
  #pragma unroll
      for (int q = 0; q < kMmatE; ++q) sh[q] = err[q] = 0.0f;
  #pragma unroll 4
      for (int j = 0; j < n; ++j) {
        const float2 b = Ts[j * 64];
        const float4 ga = *reinterpret_cast<const float4 *>(Gs + j * np);
        const float4 gb = *reinterpret_cast<const float4 *>(Gs + j * np + 2);
        const float gh[kMmatE] = {ga.x, ga.z, gb.x, gb.z}, gl[kMmatE] = {ga.y, ga.w, gb.y, gb.w};
  #pragma unroll
        for (int q = 0; q < kMmatE; ++q) {
          const fdw p = two_prod(gh[q], b.x);
          const fdw r = two_sum(sh[q], p.hi);
          sh[q] = r.hi;
          err[q] = __fadd_rn(err[q], __fadd_rn(r.lo, __fadd_rn(p.lo, __fmaf_rn(gh[q], b.y, __fmul_rn(gl[q], b.x)))));
        }
      }
  #pragma unroll
      for (int q = 0; q < kMmatE; ++q) {
        const int e = e0 + q;
        if (e >= (up ? n : nd)) continue;
        const fdw r = fast_two_sum(sh[q], err[q]);
        const size_t o = ((size_t)w * N + (up ? e : n + e)) * L + c0 + c;
        mbuf[o] = r.hi;
        mlo[o] = r.lo;
      }
    }
}
};
__global__ void __launch_bounds__(256) k_mmat_dw(DevSystem s, const double *__restrict__ ginv64,
                                                 const float *__restrict__ bt, const float *__restrict__ bt_lo,
                                                 const float *__restrict__ a_up, const float *__restrict__ a_lo,
                                                 float *__restrict__ mbuf, float *__restrict__ mlo) {
  MmatDw::run(s, ginv64, bt, bt_lo, a_up, a_lo, mbuf, mlo, blockIdx, gridDim);
}

cudaError_t launch_mmat_dw(const DevSystem &s, const double *ginv64, const float *bt, const float *bt_lo,
                           const float *a_up, const float *a_lo, float *mbuf, float *mlo, int W, cudaStream_t st) {
  if (W <= 0) return cudaSuccess;
  const int n = s.n_up, np = (n + kMmatE - 1) / kMmatE * kMmatE;
  const size_t smem = (size_t)(2 * n * np + 2 * n * 64) * sizeof(float2);
  if (smem > kMmatSmemMax) return cudaErrorInvalidValue;
  dim3 grid((s.L + 63) / 64, W);
  return launch_or_record<MmatDw, 256>(k_mmat_dw, grid, dim3(256), smem, st, s, ginv64, bt, bt_lo, a_up, a_lo, mbuf,
                                       mlo);
}

cudaError_t launch_mmat(const DevSystem &s, const double *ginv, const double *bt, const double *a_up, double *mbuf, int W,
                        cudaStream_t st) {
  if (W <= 0) return cudaSuccess;
  const int n = s.n_up;
  const size_t smem = (size_t)(n * n + 2 * n * 64) * sizeof(double);
  if (smem > kMmatSmemMax) {
    dim3 grid((s.L + 63) / 64, (n + 63) / 64 + (s.n_dn + 63) / 64, W);
    return launch_or_record<MmatTiled, 256>(k_mmat_tiled, grid, dim3(256), 0, st, s, ginv, bt, a_up, mbuf);
  }
  dim3 grid((s.L + 63) / 64, W);
  return launch_or_record<Mmat, 256>(k_mmat, grid, dim3(256), smem, st, s, ginv, bt, a_up, mbuf);
}

// the kernels of this file raise their shared-memory limit when first
// launched (launch_or_record)
cudaError_t setup_kernel_attributes() { return cudaSuccess; }

}  // namespace jagp
