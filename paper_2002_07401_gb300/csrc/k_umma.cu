// k_umma.cu -- the dense lambda contraction on the 5th-generation tensor cores
// (tcgen05.mma kind::f16, BF16 operands, FP32 accumulator in tensor memory),
// fed by TMA through a multi-stage mbarrier pipeline.
//
// Plain mode:  C[m][n] = sum_p sum_k A[m][a_p Kp + k] * B[n][b_p Kp + k]
// A holds up to four BF16 "terms" of each row side by side (each Kp wide, Kp a
// multiple of 64); B likewise.  All pairs accumulate into one FP32 tensor-
// memory accumulator.
//
// Fixed-point mode (row exponents ea[m], column exponents eb[n] given): the
// terms are 8-bit integer slices of rows scaled by powers of two,
//   a = 2^(ea - 7) (t0 + t1 / 256 + t2 / 256^2 + ...),  |t_i| <= 128,
// (exact in BF16), so every slice product is an integer below 2^14 and the
// tensor cores sum them exactly while partial sums stay below 2^24.  Pairs of
// equal weight d = a_p + b_p share an accumulator S_d (up to eight), and the
// epilogue forms C = 2^(ea + eb - 14) (S_0 + S_1 / 256 + S_2 / 256^2 + ...) as
// an unevaluated two-float sum: products of two-float rows far beyond FP32
// accuracy, which the lossy FP32 accumulation inside the tensor cores would
// not give.
//
// Two kernels.  k_umma_gemm takes any list of slice pairs: one CTA per 128 x BN
// tile, stages of one A and one B slice of a 64-wide K chunk, pair after pair.
// k_umma_tri takes the full triangle of pairs (a + b < NS) that every product
// of the library uses; see there.  Every wait is bounded by the global timer; a
// timeout sets *err.
#include <cuda.h>
#include <cuda_bf16.h>

#include <atomic>
#include <mutex>

#include "jagp_group.cuh"
#include "jagp_launch.h"

namespace jagp {

namespace {

constexpr uint64_t kWaitLimitNs = 2000000000ull;  // 2 s per wait
constexpr int kGroupM = 8;                         // row tiles per group of the tile order

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// wait for the phase with the given parity to complete; false after the limit
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  while (!mbar_try_wait(bar, parity))
    if (global_ns() - t0 > kWaitLimitNs) return false;
  return true;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

// Shared-memory matrix descriptor of a K-major tile written by TMA with the
// swizzle of its row width: rows of 128, 64 or 32 bytes (K chunks of 64, 32 or
// 16 BF16 elements), 8-row groups 8 row widths apart; the PTX layout codes of
// the 128-, 64- and 32-byte swizzles are 2, 4 and 6.
__device__ __forceinline__ uint64_t desc_kmajor(uint32_t saddr, uint32_t row_bytes) {
  const uint64_t layout = row_bytes == 128 ? 2 : (row_bytes == 64 ? 4 : 6);
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);      // start address
  d |= static_cast<uint64_t>(1) << 16;                      // leading byte offset (unused here)
  d |= static_cast<uint64_t>((8u * row_bytes) >> 4) << 32;  // stride byte offset
  d |= static_cast<uint64_t>(1) << 46;                      // descriptor version for tcgen05
  d |= layout << 61;                                        // swizzle
  return d;
}

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}

// tensor maps read from global memory (the grouped launches keep them with
// their arguments there): order the generic-proxy writes that placed them
// before their use by the tensor-map proxy.  Kernel-parameter maps need nothing.
__device__ __forceinline__ void tensormap_acquire(const CUtensorMap *a, const CUtensorMap *b) {
  if (__isGlobal(a)) asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(a) : "memory");
  if (__isGlobal(b)) asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(b) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

struct UmmaArgs {
  int m_max;             // rows the grid covers
  const int *m_dev;      // live row count on the device, or null (= m_max)
  int n;                 // output columns
  int kp;                // K per term, multiple of 64
  int bn;                // output columns per CTA (multiple of 16, <= 256)
  int stages;
  int npairs;
  int pair_a[kMaxPairs], pair_b[kMaxPairs], pair_group[kMaxPairs];
  int ngroups;           // accumulators (1 in plain mode)
  const int *a_exp;      // fixed-point mode: row exponents [m_max], else null
  const int *b_exp;      // fixed-point mode: column exponents [n]
  uint32_t idesc;
  uint32_t tmem_cols;    // power of two >= max(32, bn)
  float *out;
  float *out_lo;         // fixed-point mode: low part of a two-float result, or null
  long long ldo;         // output row pitch (elements)
  const int *out_rows;   // destination row of row m, or null (= m)
  int *err;
};

struct UmmaGemm {
  static __device__ __forceinline__ void run(const CUtensorMap &tmA, const CUtensorMap &tmB, const UmmaArgs &g,
                                             const uint3 bid, const uint3 gdim) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int M = g.m_dev ? *g.m_dev : g.m_max;
    // grouped tile order: CTAs in launch order walk kGroupM row tiles of one
    // column tile before the next column tile, so that a wave reuses both A and
    // B tiles from L2 (with large K the operands exceed L2)
    int tile_y, tile_x;
    {
      const int tiles_n = gdim.x, tiles_m = gdim.y;
      const int pid = bid.x + bid.y * tiles_n;
      const int span = kGroupM * tiles_n;
      const int first = (pid / span) * kGroupM;
      const int gsize = tiles_m - first < kGroupM ? tiles_m - first : kGroupM;
      const int r = pid - (pid / span) * span;
      tile_y = first + r % gsize;
      tile_x = r / gsize;
    }
    const int m0 = tile_y * 128;
    if (m0 >= M) return;  // whole CTA, before any barrier or tensor-memory use
    const int n0 = tile_x * g.bn;
    const uint32_t a_bytes = 128u * 128u;
    const uint32_t b_bytes = static_cast<uint32_t>(g.bn) * 128u;
    const uint32_t stage_bytes = a_bytes + b_bytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + g.stages * stage_bytes);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * g.stages + 1);
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8u * g.stages, done = full0 + 16u * g.stages;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
      for (int s = 0; s < g.stages; ++s) {
        mbar_init(full0 + 8u * s, 1);
        mbar_init(empty0 + 8u * s, 1);
      }
      mbar_init(done, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(g.tmem_cols)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int kchunks = g.kp / 64;
    const int iters = g.npairs * kchunks;
    const uint32_t tiles = smem_u32(smem);

    if (warp == 0 && lane == 0) tensormap_acquire(&tmA, &tmB);
    if (warp == 0 && lane == 0) {
      // producer: one A tile (128 x 64) and one B tile (bn x 64) per stage
      for (int it = 0; it < iters; ++it) {
        const int s = it % g.stages;
        const uint32_t use = static_cast<uint32_t>(it / g.stages);
        if (it >= g.stages && !mbar_wait(empty0 + 8u * s, (use & 1u) ^ 1u)) {
          atomicExch(g.err, 1);
          break;
        }
        const uint32_t full = full0 + 8u * s;
        mbar_expect_tx(full, stage_bytes);
        const int p = it / kchunks, c = it - p * kchunks;
        tma_load_2d(tiles + s * stage_bytes, &tmA, g.pair_a[p] * g.kp + c * 64, m0, full);
        tma_load_2d(tiles + s * stage_bytes + a_bytes, &tmB, g.pair_b[p] * g.kp + c * 64, n0, full);
      }
    } else if (warp == 1 && lane == 0) {
      // MMA issuer: four K = 16 slices per 64-wide chunk, accumulating in TMEM
      uint32_t started = 0;  // bit g: accumulator g has received its first product
      for (int it = 0; it < iters; ++it) {
        const int s = it % g.stages;
        const uint32_t use = static_cast<uint32_t>(it / g.stages);
        if (!mbar_wait(full0 + 8u * s, use & 1u)) {
          atomicExch(g.err, 2);
          break;
        }
        tc_fence_after();
        const uint32_t a0 = tiles + s * stage_bytes, b0 = a0 + a_bytes;
        const int grp = g.pair_group[it / kchunks];
        const uint32_t d_tmem = tmem + static_cast<uint32_t>(grp * g.bn);
  #pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          umma_bf16(d_tmem, desc_kmajor(a0 + kk * 32, 128u), desc_kmajor(b0 + kk * 32, 128u), g.idesc,
                    (started >> grp) & 1u);
          started |= 1u << grp;
        }
        umma_commit(empty0 + 8u * s);
      }
      umma_commit(done);  // arrives once every MMA issued above has completed
    }
    __syncwarp();

    // epilogue: tensor memory -> registers -> FP32 rows
    const bool ready = __all_sync(0xffffffffu, mbar_wait(done, 0));  // warp-uniform for tcgen05.ld
    tc_fence_after();
    if (ready) {
      const int row = m0 + warp * 32 + lane;
      const bool live = row < M;
      const long long dst = live ? (g.out_rows ? g.out_rows[row] : row) : 0;
      const long long obase = dst * g.ldo;  // element offset of this row's column 0
      const uint32_t t_row = tmem + (static_cast<uint32_t>(warp * 32) << 16);
      const int ea = (g.a_exp && live) ? g.a_exp[row] : 0;
      for (int c = 0; c < g.bn; c += 16) {
        float v[16];
        tmem_ld16(t_row + static_cast<uint32_t>(c), v);
        if (g.a_exp) {
          // v = S_0 + S_1 / 256 + S_2 / 256^2 + ... as an unevaluated sum
          // hi + lo of FP32 numbers: every S_d is an exact integer below 2^24 and
          // each addition goes through an error-free transformation (TwoSum)
          float lo[16];
  #pragma unroll
          for (int j = 0; j < 16; ++j) lo[j] = 0.0f;
          float scale = 1.0f;
          for (int q = 1; q < g.ngroups; ++q) {
            float u[16];
            tmem_ld16(t_row + static_cast<uint32_t>(q * g.bn + c), u);
            scale *= 0.00390625f;
  #pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float b = __fmul_rn(u[j], scale);  // exact: power-of-two scaling
              const float s = __fadd_rn(v[j], b);
              const float z = __fsub_rn(s, v[j]);
              const float e = __fadd_rn(__fsub_rn(v[j], __fsub_rn(s, z)), __fsub_rn(b, z));
              v[j] = s;
              lo[j] = __fadd_rn(lo[j], e);
            }
          }
  #pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float hi = __fadd_rn(v[j], lo[j]);
            const float l2 = __fsub_rn(lo[j], __fsub_rn(hi, v[j]));
            const int col = n0 + c + j;
            const int sh = ea + (col < g.n ? g.b_exp[col] : 0) - 14;
            v[j] = ldexpf(hi, sh);
            lo[j] = ldexpf(l2, sh);
          }
          if (live && g.out_lo) {
            float *ol = g.out_lo + obase;
  #pragma unroll
            for (int j = 0; j < 16; ++j)
              if (n0 + c + j < g.n) ol[n0 + c + j] = lo[j];
          }
        }
        if (live) {
          float *o = g.out + obase;
  #pragma unroll
          for (int j = 0; j < 16; ++j)
            if (n0 + c + j < g.n) o[n0 + c + j] = v[j];
        }
      }
    } else if (lane == 0) {
      atomicExch(g.err, 3);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
      tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(g.tmem_cols) : "memory");
    }
}
};

__global__ void __launch_bounds__(128) k_umma_gemm(const __grid_constant__ CUtensorMap tmA,
                                                   const __grid_constant__ CUtensorMap tmB,
                                                   const __grid_constant__ UmmaArgs g) {
  UmmaGemm::run(tmA, tmB, g, blockIdx, gridDim);
}

// ---------------------------------------------------------------------------
// k_umma_tri: the fixed-point product with every pair a + b < NS of NS slices.
//
// What bounds it: each 128 x 64 x 16 MMA takes 32 clocks of the tensor pipe but
// reads 4 KB of A and 2 KB of B from shared memory (48 clocks), so one MMA per
// pair is bound by operand reads.  The B slices of a K chunk are stacked in
// shared memory, and accumulator d sits bn tensor-memory columns after
// accumulator d - 1, so the pairs (a, 0) .. (a, NS - 1 - a) of one A slice are ONE
// product of that slice with the stacked B slices into consecutive
// accumulators: 6 A slices give 8 MMAs of up to 256 columns per K = 16 step
// instead of 21 of 64, and A is read 8 times instead of 21.
//
// Persistent CTAs (one per SM: warp 0 TMA, warp 1 MMA, eight epilogue warps)
// walk the tiles, so that the next tile's operands load during the epilogue.
// Only the K chunks in which the B tile has a non-zero element are visited
// (krange: [first, last) per 16 rows of B, found when lambda is sliced): zeros
// change no exact sum, so a banded pairing matrix costs its band, and the
// padding of K costs nothing.
// Every CTA loads its own slices, from L2: pairs of CTAs that shared a row tile's A
// slices were no faster (sweeps of 4096 walkers of 16 He 2.58 ms either way) and
// slower where column tiles are few (509 walkers of 43 + 40 electrons 5.12 against
// 4.61 ms: a pair waits for both epilogues, and an odd tile count leaves a CTA idle).
//
// TMEM: NS accumulators of bn <= 512 / NS columns.  The CTA asks for more than
// half of the SM's shared memory, so that two CTAs never wait for each other's
// tensor memory.
//
// Measured against one MMA per pair in CTA-per-tile launches: the six-slice
// lambda products of the accepted rows of 4096 walkers (about 30 thousand rows,
// K = N = 320) 403 -> 120 us (1.06 PFLOP/s of slice products); seven slices, 2048
// walkers, FP64 result 443 -> 136 us; the six products of a 512-electron sweep
// (64 walkers, K = N = 4096, a tenth of lambda non-zero) 39.3 -> 4.0 ms.
// ---------------------------------------------------------------------------
constexpr int kTriThreads = 320;
constexpr int kTriEpiWarps = 8;

struct TriArgs {
  int m_max;             // rows the grid covers
  const int *m_dev;      // live row count on the device, or null (= m_max)
  int n, bn, tiles_n;    // output columns, columns per CTA, column tiles
  int kp, klive;         // K per slice (row pitch of a slice), elements that may be non-zero
  int cw, stages;        // K chunk width in elements (64, 32, 16), chunks in flight
  const int2 *krange;    // non-zero K range per 16 rows of B, or null (= [0, klive))
  int slice_bits;
  int batch_rows, tiles_per_batch, b_batch_rows;  // batched mode (batch_rows > 0): block b of A against block b of B
  const int *a_exp, *b_exp;
  float *out, *out_lo;
  double *out64;
  long long ldo;
  const int *out_rows;
  long long o_bstride, o_rstride, o_cstride;
  int vec;               // output rows take 32-byte stores
  int add;               // out64 += (scalar stores)
  int *err;
};

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// sixteen columns of this warp's lanes; valid after tmem_ld_wait
__device__ __forceinline__ void tmem_ld16_async(uint32_t taddr, uint32_t r[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

// v * 2^sh, rounded once: by the factor 2^sh where that is a normal number
__device__ __forceinline__ float scale_pow2(float v, int sh) {
  return sh >= -126 && sh <= 127 ? __fmul_rn(v, __int_as_float((sh + 127) << 23)) : ldexpf(v, sh);
}
__device__ __forceinline__ double scale_pow2(double v, int sh) {
  const long long b = __double_as_longlong(v);
  const int e = static_cast<int>((b >> 52) & 0x7ff);
  return e > 0 && e < 0x7ff && e + sh > 0 && e + sh < 0x7ff ? __longlong_as_double(b + (static_cast<long long>(sh) << 52))
                                                            : ldexp(v, sh);
}
// an integer |x| < 2^51 as FP64 (one FP64 instruction)
__device__ __forceinline__ double small_int_to_double(long long x) {
  return __longlong_as_double(0x4338000000000000LL + x) - 6755399441055744.0;
}

__device__ __forceinline__ void store8(float *p, const float *v) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}
__device__ __forceinline__ void store4(double *p, const double *v) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3])
               : "memory");
}

template <int NS, bool F64>
struct UmmaTri {
  static __device__ __forceinline__ void run(const CUtensorMap &tmA, const CUtensorMap &tmB, const TriArgs &g,
                                             const uint3 bid, const uint3 gdim) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int M = g.m_dev ? *g.m_dev : g.m_max;
    const int tiles_m = g.batch_rows ? (g.m_max / g.batch_rows) * g.tiles_per_batch : (M + 127) / 128;
    const int total = tiles_m * g.tiles_n;
    const int first = static_cast<int>(bid.x), step = static_cast<int>(gdim.x);
    if (first >= total) return;  // before any barrier or tensor-memory use
    const uint32_t row_bytes = static_cast<uint32_t>(g.cw) * 2u;
    const uint32_t a_bytes = 128u * row_bytes, b_bytes = static_cast<uint32_t>(g.bn) * row_bytes;
    const uint32_t stage_bytes = NS * (a_bytes + b_bytes);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + g.stages * stage_bytes);
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8u * g.stages, tfull = full0 + 16u * g.stages,
                   tempty = tfull + 8u;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * g.stages + 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
      for (int s = 0; s < g.stages; ++s) {
        mbar_init(full0 + 8u * s, 1);
        mbar_init(empty0 + 8u * s, 1);
      }
      mbar_init(tfull, 1);
      mbar_init(tempty, kTriEpiWarps);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(512)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t tiles = smem_u32(smem);

    // tile t: row tile, column tile
    auto place = [&](int t, int &ty, int &cx) {
      // kGroupM row tiles of one column step before the next, so that a wave
      // shares operand tiles in L2
      const int span = kGroupM * g.tiles_n, q = t / span, r = t - q * span;
      const int gsize = tiles_m - q * kGroupM < kGroupM ? tiles_m - q * kGroupM : kGroupM;
      ty = q * kGroupM + r % gsize;
      cx = r / gsize;
    };
    // K chunks [c0, c1) of a column tile
    auto chunks = [&](int cx, int &c0, int &c1) {
      int lo = 0, hi = g.klive;
      if (g.krange) {
        lo = g.kp;
        hi = 0;
        const int b0 = cx * g.bn / 16, b1 = b0 + g.bn / 16, nb = (g.n + 15) / 16;
        for (int b = b0; b < b1 && b < nb; ++b) {
          const int2 r = g.krange[b];
          lo = r.x < lo ? r.x : lo;
          hi = r.y > hi ? r.y : hi;
        }
      }
      c0 = lo / g.cw;
      c1 = (hi + g.cw - 1) / g.cw;
      if (c1 <= c0) {  // every element zero: one chunk clears the accumulators
        c0 = 0;
        c1 = 1;
      }
    };
    auto rows_of = [&](int ty, int &bb, int &bt0, int &m0) {
      bb = g.batch_rows ? ty / g.tiles_per_batch : 0;
      bt0 = g.batch_rows ? (ty - bb * g.tiles_per_batch) * 128 : 0;
      m0 = g.batch_rows ? bb * g.batch_rows + bt0 : ty * 128;
    };

    if (warp == 0) {
      if (lane == 0) {
        // producer: every slice of A and of B for one K chunk per stage
        tensormap_acquire(&tmA, &tmB);
        int it = 0;
        bool ok = true;
        for (int t = first; t < total && ok; t += step) {
          int ty, cx, c0, c1, bb, bt0, m0;
          place(t, ty, cx);
          chunks(cx, c0, c1);
          rows_of(ty, bb, bt0, m0);
          const int brow = bb * g.b_batch_rows + cx * g.bn;
          for (int c = c0; c < c1; ++c, ++it) {
            const int s = it % g.stages;
            if (it >= g.stages && !mbar_wait(empty0 + 8u * s, ((it / g.stages) & 1u) ^ 1u)) {
              atomicExch(g.err, 1);
              ok = false;
              break;
            }
            const uint32_t full = full0 + 8u * s, base = tiles + s * stage_bytes, bbase = base + NS * a_bytes;
            mbar_expect_tx(full, stage_bytes);
  #pragma unroll
            for (int a = 0; a < NS; ++a) tma_load_2d(base + a * a_bytes, &tmA, a * g.kp + c * g.cw, m0, full);
  #pragma unroll
            for (int b = 0; b < NS; ++b) tma_load_2d(bbase + b * b_bytes, &tmB, b * g.kp + c * g.cw, brow, full);
          }
        }
        // the last uses of every stage: no load is in flight when this CTA ends
        for (int u = it > g.stages ? it - g.stages : 0; u < it; ++u)
          if (!mbar_wait(empty0 + 8u * (u % g.stages), (u / g.stages) & 1u)) {
            atomicExch(g.err, 1);
            break;
          }
      }
    } else if (warp == 1) {
      if (lane == 0) {
        int it = 0, done = 0;
        bool ok = true;
        const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(128 >> 4) << 24);
        const int ksteps = g.cw / 16;
        for (int t = first; t < total && ok; t += step, ++done) {
          int ty, cx, c0, c1;
          place(t, ty, cx);
          chunks(cx, c0, c1);
          if (done > 0 && !mbar_wait(tempty, (done - 1) & 1u)) {
            atomicExch(g.err, 2);
            break;
          }
          tc_fence_after();
          for (int c = c0; c < c1; ++c, ++it) {
            const int s = it % g.stages;
            if (!mbar_wait(full0 + 8u * s, (it / g.stages) & 1u)) {
              atomicExch(g.err, 2);
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t base = tiles + s * stage_bytes;
            const uint64_t da = desc_kmajor(base, row_bytes), db = desc_kmajor(base + NS * a_bytes, row_bytes);
            for (int kk = 0; kk < ksteps; ++kk) {
              // descriptor addresses count 16-byte units
              const uint64_t ak = da + kk * 2, bk = db + kk * 2;
              const uint32_t init = (c > c0 || kk > 0) ? 1u : 0u;
  #pragma unroll
              for (int a = 0; a < NS; ++a) {
                // slice a against stacked slices 0 .. NS - 1 - a, into accumulators a .. NS - 1
                const int cols = (NS - a) * g.bn;
                const uint64_t aa = ak + a * (a_bytes >> 4);
                const uint32_t d = tmem + static_cast<uint32_t>(a * g.bn);
                const uint32_t acc = a > 0 ? 1u : init;
                const int n1 = cols < 256 ? cols : 256;
                umma_bf16(d, aa, bk, idesc0 | (static_cast<uint32_t>(n1 >> 3) << 17), acc);
                if (cols > 256)
                  umma_bf16(d + 256u, aa, bk + ((256u * row_bytes) >> 4),
                            idesc0 | (static_cast<uint32_t>((cols - 256) >> 3) << 17), acc);
              }
            }
            umma_commit(empty0 + 8u * s);
          }
          if (ok) umma_commit(tfull);
        }
      }
    } else {
      // epilogue warps 2 .. 9: tensor-memory lanes 32 (warp % 4) .. + 31 are the
      // rows, the two warps of a lane quarter take alternate 16-column groups
      const int quarter = warp & 3, half = (warp - 2) >> 2;
      const int ngrp = g.bn / 16;
      int done = 0;
      for (int t = first; t < total; t += step, ++done) {
        int ty, cx, bb, bt0, m0;
        place(t, ty, cx);
        rows_of(ty, bb, bt0, m0);
        const int n0 = cx * g.bn;
        const int r = quarter * 32 + lane, row = m0 + r;
        const bool live = row < M && (!g.batch_rows || bt0 + r < g.batch_rows);
        const long long dst = live ? (g.out_rows ? g.out_rows[row] : row) : 0;
        const long long obase =
            g.o_cstride ? (long long)bb * g.o_bstride + (long long)(bt0 + r) * g.o_rstride : dst * g.ldo;
        const long long ocs = g.o_cstride ? g.o_cstride : 1;
        const int ea = live ? g.a_exp[row] : 0;
        const int *be = g.b_exp + bb * g.b_batch_rows;
        const uint32_t t_row = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
        if (!__all_sync(0xffffffffu, mbar_wait(tfull, done & 1u))) {  // warp-uniform for tcgen05.ld
          if (lane == 0) atomicExch(g.err, 3);
          break;
        }
        tc_fence_after();
        bool released = false;
        for (int cg = half; cg < ngrp; cg += 2) {
          uint32_t u[NS][16];
  #pragma unroll
          for (int q = 0; q < NS; ++q) tmem_ld16_async(t_row + static_cast<uint32_t>(q * g.bn + cg * 16), u[q]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          // the values may be used from here on, not earlier
  #pragma unroll
          for (int q = 0; q < NS; ++q)
  #pragma unroll
            for (int j = 0; j < 16; ++j) asm volatile("" : "+r"(u[q][j]));
          if (cg + 2 >= ngrp) {  // this warp's last reads: the accumulators may be overwritten
            tc_fence_before();
            if (lane == 0) mbar_arrive(tempty);
            released = true;
          }
          const int c0 = n0 + cg * 16;
          if constexpr (F64) {
            // the exact sums as two integers of NS / 2 terms each (H leading, the
            // rest below), joined by one rounding: hi 2^(b (NS - H)) + lo
            constexpr int H = NS / 2;
            const int b = g.slice_bits;
            const double up = __longlong_as_double(static_cast<long long>(1023 + b * (NS - H)) << 52);
            const int sh0 = ea - b * (NS - 1) - 2 * (b - 1);
            double v[16];
  #pragma unroll
            for (int j = 0; j < 16; ++j) {
              long long hi = 0, lo = 0;
  #pragma unroll
              for (int q = 0; q < H; ++q) hi = hi * (1ll << b) + __float2int_rn(__uint_as_float(u[q][j]));
  #pragma unroll
              for (int q = H; q < NS; ++q) lo = lo * (1ll << b) + __float2int_rn(__uint_as_float(u[q][j]));
              double s = fma(small_int_to_double(hi), up, small_int_to_double(lo));
              // a non-finite operand shows in its leading slice's sum
              if (!(fabsf(__uint_as_float(u[0][j])) <= 3.0e38f)) s = __longlong_as_double(0x7ff8000000000000LL);
              v[j] = scale_pow2(s, sh0 + (c0 + j < g.n ? be[c0 + j] : 0));
            }
            if (live) {
              double *o = g.out64 + obase;
              if (g.add) {
  #pragma unroll
                for (int j = 0; j < 16; ++j)
                  if (c0 + j < g.n) o[(c0 + j) * ocs] += v[j];
              } else if (g.vec && c0 + 16 <= g.n) {
  #pragma unroll
                for (int j = 0; j < 16; j += 4) store4(o + c0 + j, v + j);
              } else {
  #pragma unroll
                for (int j = 0; j < 16; ++j)
                  if (c0 + j < g.n) o[(c0 + j) * ocs] = v[j];
              }
            }
          } else {
            // S_0 + S_1 / 256 + S_2 / 256^2 + ... as an unevaluated sum hi + lo of
            // FP32 numbers: every S_d is an exact integer below 2^24 and each
            // addition goes through an error-free transformation (TwoSum)
            float v[16], lo[16];
  #pragma unroll
            for (int j = 0; j < 16; ++j) {
              v[j] = __uint_as_float(u[0][j]);
              lo[j] = 0.0f;
            }
            float scale = 1.0f;
  #pragma unroll
            for (int q = 1; q < NS; ++q) {
              scale *= 0.00390625f;
  #pragma unroll
              for (int j = 0; j < 16; ++j) {
                const float b = __fmul_rn(__uint_as_float(u[q][j]), scale);  // exact: power-of-two scaling
                const float s = __fadd_rn(v[j], b);
                const float z = __fsub_rn(s, v[j]);
                const float e = __fadd_rn(__fsub_rn(v[j], __fsub_rn(s, z)), __fsub_rn(b, z));
                v[j] = s;
                lo[j] = __fadd_rn(lo[j], e);
              }
            }
  #pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float hi = __fadd_rn(v[j], lo[j]);
              const float l2 = __fsub_rn(lo[j], __fsub_rn(hi, v[j]));
              const int sh = ea + (c0 + j < g.n ? be[c0 + j] : 0) - 14;
              v[j] = scale_pow2(hi, sh);
              lo[j] = scale_pow2(l2, sh);
            }
            if (live) {
              float *o = g.out + obase, *ol = g.out_lo ? g.out_lo + obase : nullptr;
              if (g.vec && c0 + 16 <= g.n) {
                store8(o + c0, v);
                store8(o + c0 + 8, v + 8);
                if (ol) {
                  store8(ol + c0, lo);
                  store8(ol + c0 + 8, lo + 8);
                }
              } else {
  #pragma unroll
                for (int j = 0; j < 16; ++j)
                  if (c0 + j < g.n) {
                    o[(c0 + j) * ocs] = v[j];
                    if (ol) ol[(c0 + j) * ocs] = lo[j];
                  }
              }
            }
          }
        }
        if (!released) {  // a warp without columns
          tc_fence_before();
          if (lane == 0) mbar_arrive(tempty);
        }
      }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
      tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
  }
};

template <int NS, bool F64>
__global__ void __launch_bounds__(kTriThreads, 1) k_umma_tri(const __grid_constant__ CUtensorMap tmA,
                                                             const __grid_constant__ CUtensorMap tmB,
                                                             const __grid_constant__ TriArgs g) {
  UmmaTri<NS, F64>::run(tmA, tmB, g, blockIdx, gridDim);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// 2-D BF16 map with a 128-byte-swizzled box of 64 (inner) x box_rows
// box of cw x box_rows BF16 elements, swizzled by its row width (cw = 64, 32
// or 16: 128-, 64- or 32-byte rows)
bool make_map(CUtensorMap *m, const void *base, uint64_t inner, uint64_t rows, uint32_t box_rows, uint32_t cw) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {inner, rows};
  cuuint64_t strides[1] = {inner * 2};
  cuuint32_t box[2] = {cw, box_rows};
  cuuint32_t es[2] = {1, 1};
  const CUtensorMapSwizzle sw =
      cw == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : (cw == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

int umma_pick_bn(int n, int max_bn) {
  if (n <= max_bn) return ((n + 15) / 16) * 16 < 32 ? 32 : ((n + 15) / 16) * 16;
  const int tiles = (n + max_bn - 1) / max_bn;
  return (((n + tiles - 1) / tiles) + 15) / 16 * 16;
}

namespace {
int g_smem_optin = 220 * 1024;  // the kernel's dynamic shared-memory limit, set once per process

uint32_t chunk_stage_bytes(int na, int nb, int bn, int cw) {
  return (static_cast<uint32_t>(na) * 128u + static_cast<uint32_t>(nb * bn)) * static_cast<uint32_t>(cw) * 2u;
}
// K chunk width: stages_max -1, -2, -3 -> 64, 32, 16
int chunk_width(int stages_max) { return stages_max == -1 ? 64 : (stages_max == -2 ? 32 : 16); }
// room for the stages: the limit less the 1 KB alignment slack and the barriers
uint32_t chunk_budget() { return static_cast<uint32_t>(g_smem_optin - 1024 - 64); }
}  // namespace

bool umma_chunk_fits(int npairs, const int *pair_a, const int *pair_b, int bn, int stages_max) {
  int na = 0, nb = 0;
  for (int p = 0; p < npairs; ++p) {
    na = pair_a[p] + 1 > na ? pair_a[p] + 1 : na;
    nb = pair_b[p] + 1 > nb ? pair_b[p] + 1 : nb;
  }
  return 2u * chunk_stage_bytes(na, nb, bn, chunk_width(stages_max)) <= chunk_budget();
}

namespace {
// the full triangle a + b < ns of ns slices, each pair once, in any order
bool full_triangle(int npairs, const int *pair_a, const int *pair_b, int ns) {
  if (ns < 6 || ns > 8 || npairs != ns * (ns + 1) / 2) return false;
  bool seen[8][8] = {};
  for (int p = 0; p < npairs; ++p) {
    const int a = pair_a[p], b = pair_b[p];
    if (a < 0 || b < 0 || a + b >= ns || seen[a][b]) return false;
    seen[a][b] = true;
  }
  return true;
}

int sm_count() {
  static std::atomic<int> count[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 152;
  const int slot = dev >= 0 && dev < 64 ? dev : 0;
  int n = count[slot].load(std::memory_order_relaxed);
  if (n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 152;
    count[slot].store(n, std::memory_order_relaxed);
  }
  return n;
}

// K chunk width and stages of a tri tile: 32-wide chunks where three stages of
// every slice fit (64-byte TMA rows), else 16-wide ones; pinned: 64, 32 or 16 where two fit
void tri_stages(int ns, int bn, int pinned, int *cw, int *stages) {
  const uint32_t budget = chunk_budget() - 128;  // (barriers of up to eight stages)
  const uint32_t per = static_cast<uint32_t>(ns) * (128u + bn) * 2u;  // bytes per K element
  int w = pinned;
  if (w == 0 || 2 * per * w > budget) w = 3 * per * 32 <= budget ? 32 : 16;
  *cw = w;
  const uint32_t s = budget / (per * w);
  *stages = static_cast<int>(s > 8 ? 8 : s);
}

// Columns per CTA (multiple of 16, at most limit): the width with the least
// estimated time of one CTA's share.  Clocks per K = 16 step: the tensor pipe
// (bn / 2 per slice pair), the operand reads from shared memory (128 bytes a
// clock) or the loads from L2 (about 32 bytes a clock and SM), whichever is
// most; fixed clocks per tile for the epilogue and the pipeline's fill.
int tri_tile(int ns, int n, int tiles_m, int klive, int limit) {
  const int sms = sm_count();
  double best = 0.0;
  int bn = 16;
  for (int w = 16; w <= limit; w += 16) {
    int reads = 0;  // A slice reads per step
    for (int a = 0; a < ns; ++a) reads += (ns - a) * w > 256 ? 2 : 1;
    const double pairs = 0.5 * ns * (ns + 1), math = pairs * w / 2, smem = (reads * 4096.0 + pairs * w * 32) / 128;
    const double l2 = ns * 32.0 * (128.0 + w) / 32;
    double t = math > smem ? math : smem;
    if (l2 > t) t = l2;
    const long long tiles = (long long)tiles_m * ((n + w - 1) / w);
    const double share = static_cast<double>((tiles + sms - 1) / sms);
    const double cost = share * (t * ((klive + 15) / 16) + 1500.0 + 40.0 * w);
    if (best == 0.0 || cost < best) {
      best = cost;
      bn = w;
    }
  }
  return bn;
}

template <int NS, bool F64>
cudaError_t launch_tri(const CUtensorMap &ta, const CUtensorMap &tb, const TriArgs &g, int grid, size_t smem,
                       cudaStream_t st) {
  return launch_or_record<UmmaTri<NS, F64>, kTriThreads>(k_umma_tri<NS, F64>, dim3(grid), dim3(kTriThreads), smem, st,
                                                         ta, tb, g);
}
}  // namespace

cudaError_t launch_umma_gemm(const uint16_t *A, int m_max, const int *m_dev, int a_terms, const uint16_t *B, int n,
                             int b_terms, int kp, int npairs, const int *pair_a, const int *pair_b, float *out,
                             long long ldo, const int *out_rows, int *err, cudaStream_t st, const int *a_exp,
                             const int *b_exp, float *out_lo, int bn_max, double *out64, int slice_bits,
                             int batch_rows, int batches, int stages_max, int b_batch_rows, long long o_bstride,
                             long long o_rstride, long long o_cstride, const int2 *krange, int klive,
                             bool add) {
  if (m_max <= 0 || n <= 0) return cudaSuccess;
  if (kp <= 0 || kp % 64 != 0 || npairs < 1 || npairs > kMaxPairs || a_terms < 1 || b_terms < 1)
    return cudaErrorInvalidValue;
  if (out64 && (!a_exp || (slice_bits != 7 && slice_bits != 8))) return cudaErrorInvalidValue;
  if ((reinterpret_cast<uintptr_t>(A) & 15u) || (reinterpret_cast<uintptr_t>(B) & 15u)) return cudaErrorInvalidValue;
  if ((a_exp == nullptr) != (b_exp == nullptr)) return cudaErrorInvalidValue;
  if (bn_max < 0 || bn_max % 16) return cudaErrorInvalidValue;
  for (int p = 0; p < npairs; ++p)
    if (pair_a[p] < 0 || pair_a[p] >= a_terms || pair_b[p] < 0 || pair_b[p] >= b_terms) return cudaErrorInvalidValue;
  CUtensorMap ta, tb;
  if (a_exp && a_terms == b_terms && full_triangle(npairs, pair_a, pair_b, a_terms) && (out64 || a_terms == 6)) {
    TriArgs g{};
    if (b_batch_rows <= 0) b_batch_rows = batch_rows;
    if (batch_rows < 0 || (batch_rows > 0 && (batches <= 0 || n > b_batch_rows))) return cudaErrorInvalidValue;
    if (o_cstride != 0 && (batch_rows <= 0 || out_rows)) return cudaErrorInvalidValue;
    if (stages_max < -3) return cudaErrorInvalidValue;
    g.m_max = m_max;
    g.m_dev = m_dev;
    g.n = n;
    g.kp = kp;
    g.klive = klive > 0 && klive < kp ? klive : kp;
    g.batch_rows = batch_rows;
    g.b_batch_rows = b_batch_rows;
    g.tiles_per_batch = batch_rows > 0 ? (batch_rows + 127) / 128 : 0;
    const int tiles_m = batch_rows > 0 ? batches * g.tiles_per_batch : (m_max + 127) / 128;
    // as many columns as NS accumulators leave room for in 512 (80 of six, 64
    // of seven or eight), or the pinned width (64 stands for the widest)
    const int widest = a_terms == 6 ? 80 : 64;
    g.bn = tri_tile(a_terms, n, tiles_m, g.klive, bn_max > 0 && bn_max < 64 ? bn_max : widest);
    tri_stages(a_terms, g.bn, stages_max < 0 ? chunk_width(stages_max) : 0, &g.cw, &g.stages);
    g.tiles_n = (n + g.bn - 1) / g.bn;
    g.krange = krange;
    g.slice_bits = slice_bits;
    g.a_exp = a_exp;
    g.b_exp = b_exp;
    g.out = out;
    g.out_lo = out_lo;
    g.out64 = out64;
    g.ldo = ldo;
    g.out_rows = out_rows;
    g.o_bstride = o_bstride;
    g.o_rstride = o_rstride;
    g.o_cstride = o_cstride;
    g.err = err;
    g.add = add && out64;
    const long long unit = out64 ? 4 : 8;  // elements of a 32-byte store
    const uintptr_t bases = out64 ? reinterpret_cast<uintptr_t>(out64)
                                  : reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(out_lo);
    g.vec = bases % 32 == 0 && (o_cstride ? o_cstride == 1 && o_bstride % unit == 0 && o_rstride % unit == 0
                                          : ldo % unit == 0);
    const uint64_t rows_b = batch_rows > 0 ? static_cast<uint64_t>(b_batch_rows) * batches : static_cast<uint64_t>(n);
    if (!make_map(&ta, A, static_cast<uint64_t>(a_terms) * kp, static_cast<uint64_t>(m_max), 128,
                  static_cast<uint32_t>(g.cw)) ||
        !make_map(&tb, B, static_cast<uint64_t>(b_terms) * kp, rows_b, static_cast<uint32_t>(g.bn),
                  static_cast<uint32_t>(g.cw)))
      return cudaErrorInvalidValue;
    size_t smem = 1024 + static_cast<size_t>(g.stages) * a_terms * (128 + g.bn) * g.cw * 2 + 8 * (2 * g.stages + 2) + 16;
    if (smem < 120 * 1024) smem = 120 * 1024;  // one CTA per SM (see the kernel)
    const long long tiles = (long long)tiles_m * g.tiles_n;
    const int sms = sm_count();
    const int grid = static_cast<int>(tiles < sms ? tiles : sms);
    if (!out64) return launch_tri<6, false>(ta, tb, g, grid, smem, st);
    if (a_terms == 6) return launch_tri<6, true>(ta, tb, g, grid, smem, st);
    if (a_terms == 7) return launch_tri<7, true>(ta, tb, g, grid, smem, st);
    return launch_tri<8, true>(ta, tb, g, grid, smem, st);
  }
  // any other list of pairs: FP32 (or two-float) rows, no batches
  if (out64 || batch_rows != 0 || o_cstride != 0) return cudaErrorInvalidValue;
  UmmaArgs g{};
  g.ngroups = 1;
  for (int p = 0; p < npairs; ++p) {
    g.pair_a[p] = pair_a[p];
    g.pair_b[p] = pair_b[p];
    g.pair_group[p] = a_exp ? pair_a[p] + pair_b[p] : 0;  // fixed-point mode: the accumulator of weight 256^-(a + b)
    if (g.pair_group[p] >= 8) return cudaErrorInvalidValue;
    if (g.pair_group[p] + 1 > g.ngroups) g.ngroups = g.pair_group[p] + 1;
  }
  g.a_exp = a_exp;
  g.b_exp = b_exp;
  g.m_max = m_max;
  g.m_dev = m_dev;
  g.n = n;
  g.kp = kp;
  // the ngroups accumulators of bn columns share the 512 tensor-memory columns;
  // bn_max (a multiple of 16) may lower the limit
  int limit = g.ngroups <= 2 ? 256 : (g.ngroups <= 4 ? 128 : (g.ngroups <= 5 ? 96 : 64));
  if (bn_max > 0) limit = bn_max < limit ? bn_max : limit;
  g.bn = umma_pick_bn(n, limit);
  const uint32_t stage_bytes = 128u * 128u + static_cast<uint32_t>(g.bn) * 128u;
  // pipeline depth: as many stages as fit in 200 KB, at most 6
  g.stages = static_cast<int>((200u * 1024u) / stage_bytes);
  if (g.stages > 6) g.stages = 6;
  g.npairs = npairs;
  g.idesc = (1u << 4)                                   // D: FP32
            | (1u << 7) | (1u << 10)                    // A, B: BF16
            | (static_cast<uint32_t>(g.bn >> 3) << 17)  // N
            | (static_cast<uint32_t>(128 >> 4) << 24);  // M
  uint32_t cols = 32;
  while (cols < static_cast<uint32_t>(g.bn * g.ngroups)) cols <<= 1;
  if (cols > 512) return cudaErrorInvalidValue;
  g.tmem_cols = cols;
  g.out = out;
  g.out_lo = a_exp ? out_lo : nullptr;
  g.ldo = ldo;
  g.out_rows = out_rows;
  g.err = err;
  if (!make_map(&ta, A, static_cast<uint64_t>(a_terms) * kp, static_cast<uint64_t>(m_max), 128, 64) ||
      !make_map(&tb, B, static_cast<uint64_t>(b_terms) * kp, static_cast<uint64_t>(n), static_cast<uint32_t>(g.bn), 64))
    return cudaErrorInvalidValue;
  const size_t smem = 1024 + static_cast<size_t>(g.stages) * stage_bytes + 8 * (2 * g.stages + 1) + 16;
  dim3 grid((n + g.bn - 1) / g.bn, (m_max + 127) / 128);
  return launch_or_record<UmmaGemm, 128>(k_umma_gemm, grid, dim3(128), smem, st, ta, tb, g);
}

// ---------------------------------------------------------------------------
// Fixed-point operand packing.  Operand rows are compacted in list order: row
// m comes from table row list[m] (m < *count) or, without a list, from
// (m / nsub) * stride + m % nsub (m < nrows); rows_out[m] records it so that
// the contraction can write its result row back in place.  One warp per row.
// Each FP32 row is scaled by
// 2^-e (e = 1 + the binary exponent of its largest magnitude) and cut into
// kFixedSlices exact 8-bit integer slices t0, t1, ... (|t| <= 128), stored as
// BF16 side by side, with e in exps[m].  Every step of the cut is exact in
// FP32.  A two-float row P + P_lo is cut the same way, its remainder carried
// from slice to slice as an exact two-float sum (TwoSum), so that the slices
// take the low part's bits as well.  A_at / exps_at (or null) receive the same
// slices and exponent at the table row's own place (the refresh's operands,
// kept current row by row as moves are accepted); A null writes only those.
// ---------------------------------------------------------------------------
struct PackFixed {
  static __device__ __forceinline__ void run(const float *__restrict__ P, const float *__restrict__ P_lo,
                                             const int *__restrict__ list, const int *__restrict__ count, int nrows,
                                             int nsub, int stride, int L, int kp, uint16_t *__restrict__ A,
                                             int *__restrict__ rows_out, int *__restrict__ exps,
                                             uint16_t *__restrict__ A_at, int *__restrict__ exps_at, const uint3 bid,
                                             const uint3 gdim) {
    assume_global(P);
    const int rows = count ? *count : nrows;
    const int lane = threadIdx.x & 31;
    const long nw = (long)gdim.x * (blockDim.x >> 5);
    for (long m = (long)bid.x * (blockDim.x >> 5) + (threadIdx.x >> 5); m < rows; m += nw) {
      const long phys = list ? (long)list[m] : (m / nsub) * stride + (m % nsub);
      const float *src = P + phys * L;
      const float *srl = P_lo ? P_lo + phys * L : nullptr;
      float mx = 0.0f;
      for (int k = lane; k < L; k += 32) mx = fmaxf(mx, fabsf(src[k]));
  #pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const int e = (mx > 0.0f) ? ilogbf(mx) + 1 : 0;
      if (lane == 0) {
        if (A) {
          rows_out[m] = (int)phys;
          exps[m] = e;
        }
        if (exps_at) exps_at[phys] = e;
      }
      uint16_t *dst = A ? A + m * kFixedSlices * (long)kp : nullptr;
      uint16_t *at = A_at ? A_at + phys * kFixedSlices * (long)kp : nullptr;
      // two consecutive elements per lane
      for (int k = 2 * lane; k < kp; k += 64) {
        float x[2], xl[2];
  #pragma unroll
        for (int h = 0; h < 2; ++h) {
          const bool in = k + h < L;
          x[h] = in ? scale_pow2(src[k + h], 7 - e) : 0.0f;             // |x| < 128
          xl[h] = in && srl ? scale_pow2(srl[k + h], 7 - e) : 0.0f;     // the low part, in the same scale
        }
  #pragma unroll
        for (int t = 0; t < kFixedSlices; ++t) {
          uint32_t v = 0;
  #pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float q = rintf(x[h]);
            // a small integer's BF16 bits: the leading half of its FP32 number
            v |= (__float_as_uint(q) >> 16) << (16 * h);
            const fdw r = two_sum(__fsub_rn(x[h], q), xl[h]);  // remainder + low part, exactly
            x[h] = __fmul_rn(r.hi, 256.0f);
            xl[h] = __fmul_rn(r.lo, 256.0f);
          }
          if (dst) *reinterpret_cast<uint32_t *>(dst + t * kp + k) = v;
          if (at) *reinterpret_cast<uint32_t *>(at + t * kp + k) = v;
        }
      }
    }
}
};
__global__ void __launch_bounds__(256) k_pack_fixed(const float *__restrict__ P, const float *__restrict__ P_lo,
                                                    const int *__restrict__ list, const int *__restrict__ count,
                                                    int nrows, int nsub, int stride, int L, int kp,
                                                    uint16_t *__restrict__ A, int *__restrict__ rows_out,
                                                    int *__restrict__ exps, uint16_t *__restrict__ A_at,
                                                    int *__restrict__ exps_at) {
  PackFixed::run(P, P_lo, list, count, nrows, nsub, stride, L, kp, A, rows_out, exps, A_at, exps_at, blockIdx,
                 gridDim);
}

cudaError_t launch_pack_fixed(const float *P, const float *P_lo, const int *list, const int *count, int nrows,
                              int nsub, int stride, int L, int kp, uint16_t *A, int *rows_out, int *exps,
                              int max_rows, cudaStream_t st, uint16_t *A_at, int *exps_at) {
  if (max_rows <= 0) return cudaSuccess;
  long blocks = (max_rows + 7) / 8;
  if (blocks > 152 * 16) blocks = 152 * 16;
  return launch_or_record<PackFixed, 256>(k_pack_fixed, dim3((int)blocks), dim3(256), 0, st, P, P_lo, list, count,
                                          nrows, nsub > 0 ? nsub : 1, stride, L, kp, A, rows_out, exps, A_at, exps_at);
}

// An FP64 value v, |v| < 2^e, as NSL slices of BITS bits: the integer nearest to
// v 2^(NSL BITS - 1 - e) cut from the top, each slice the nearest integer
// (|t| <= 2^(BITS - 1), exact in BF16).  Integer instructions only: as FP64
// arithmetic (scale, round, subtract, multiply per slice) the cut was bound by
// the FP64 pipe, which takes 16 clocks per warp instruction.  A value that is not
// finite gives NaN slices.
template <int NSL, int BITS>
__device__ __forceinline__ void cut_slices(double v, int e, uint16_t t[NSL]) {
  const long long b = __double_as_longlong(v);
  const int ef = static_cast<int>((b >> 52) & 0x7ff);
  long long m = b & 0xfffffffffffffll;
  if (ef) m |= 1ll << 52;
  // v = +-m 2^(max(ef, 1) - 1075); shift to units of 2^(e + 1 - NSL BITS)
  const int sh = (ef ? ef : 1) - 1075 + NSL * BITS - 1 - e;
  if (sh >= 0) {
    m <<= sh < 10 ? sh : 10;  // |v| < 2^e leaves at most 55 bits
  } else {
    const int r = -sh;
    m = r > 54 ? 0 : (m + (1ll << (r - 1))) >> r;
  }
  if (b < 0) m = -m;
#pragma unroll
  for (int q = 0; q < NSL; ++q) {
    constexpr int kLast = (NSL - 1) * BITS;
    const int s = kLast - q * BITS;
    const int d = static_cast<int>(s ? (m + (1ll << (s ? s - 1 : 0))) >> s : m);
    m -= static_cast<long long>(d) << s;
    // a small integer's BF16 bits: the leading half of its FP32 number
    t[q] = ef == 0x7ff ? static_cast<uint16_t>(0x7fc0)
                       : static_cast<uint16_t>(__float_as_uint(__int_as_float(0x4B400000 + d) - 12582912.0f) >> 16);
  }
}
// the exponent e with |v| < 2^e from the largest leading word of |v| (0 where a
// value is not finite: the products are then NaN whatever the scale)
__device__ __forceinline__ unsigned abs_hi(double v) {
  return static_cast<unsigned>(static_cast<unsigned long long>(__double_as_longlong(v)) >> 32) & 0x7fffffffu;
}
__device__ __forceinline__ int exponent_of(unsigned hi) {
  const int ef = static_cast<int>(hi >> 20);
  return ef == 0x7ff || hi == 0u ? 0 : (ef ? ef : 1) - 1022;
}
// the same of one value times 2^d, for a maximum over several: kNoExponent for 0,
// kNotFinite where it is not finite; then the maximum's
constexpr int kNoExponent = -0x7fffffff, kNotFinite = 0x7fffffff;
__device__ __forceinline__ int element_exponent(double v, int d) {
  const unsigned hi = abs_hi(v), lo = static_cast<unsigned>(__double2loint(v));
  return hi >= 0x7ff00000u ? kNotFinite : ((hi | lo) == 0u ? kNoExponent : exponent_of(hi | 1u) + d);
}
__device__ __forceinline__ int exponent_of_max(int e) { return e == kNotFinite || e == kNoExponent ? 0 : e; }

// ---------------------------------------------------------------------------
// Powers of two that balance a product sum_k X[k][c] Y(k, y) of exact slices.  The cut
// keeps 55 bits of a column's largest entry over k, which is what the sum needs only
// while no k is weak in X and strong in Y: an electron far from all atoms has a row of
// G~ of 1e-12, say, and entries of G~^{-1} of 1e12, beside which the others' would lose
// all their bits (local energies of 34 + 33 electrons, two of them so, were off by 19 %;
// with this 1e-12, as with FP64 instructions).  s_k <= 0: Y(k, .) is taken times 2^-s_k,
// X[k][.] times 2^s_k, so that the largest |Y(k, .)| of every k has the same exponent.
// A CTA per walker; bound by one read of Y, far below the product's operands (gradients
// of 256 walkers of 64 He: 27.7 ms with and without).
// ---------------------------------------------------------------------------
struct BalanceTerms {
  static __device__ __forceinline__ void run(const double *__restrict__ Y, int n, int K, int ny, int y_rows,
                                             int *__restrict__ s, const uint3 bid, const uint3 gdim) {
    assume_global(Y, s);
    extern __shared__ int ek[];  // [K] exponent of the largest |Y(k, .)|
    __shared__ int top[8];
    const int w = bid.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double *Yw = Y + (size_t)w * n * n;
    if (y_rows) {
      for (int k = tid; k < K; k += 256) {
        int e = kNoExponent;
#pragma unroll 4
        for (int y = 0; y < ny; ++y) e = max(e, element_exponent(Yw[(size_t)y * n + k], 0));
        ek[k] = e;
      }
    } else {
      for (int k = warp; k < K; k += 8) {
        int e = kNoExponent;
        for (int y = lane; y < ny; y += 32) e = max(e, element_exponent(Yw[(size_t)k * n + y], 0));
        e = __reduce_max_sync(0xffffffffu, e);
        if (lane == 0) ek[k] = e;
      }
    }
    __syncthreads();
    int m = kNoExponent;
    for (int k = tid; k < K; k += 256)
      if (ek[k] != kNotFinite) m = max(m, ek[k]);
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) top[warp] = m;
    __syncthreads();
    for (int q = 0; q < 8; ++q) m = max(m, top[q]);
    for (int k = tid; k < K; k += 256)
      s[(size_t)w * K + k] = ek[k] == kNotFinite || ek[k] == kNoExponent ? 0 : ek[k] - m;
  }
};
__global__ void __launch_bounds__(256) k_balance_terms(const double *__restrict__ Y, int n, int K, int ny, int y_rows,
                                                       int *__restrict__ s) {
  BalanceTerms::run(Y, n, K, ny, y_rows, s, blockIdx, gridDim);
}
cudaError_t launch_balance_terms(const double *Y, int n, int K, int ny, bool y_rows, int W, int *s, cudaStream_t st) {
  if (W <= 0 || K <= 0) return cudaSuccess;
  return launch_or_record<BalanceTerms, 256>(k_balance_terms, dim3(W), dim3(256), (size_t)K * sizeof(int), st, Y, n, K,
                                             ny, y_rows ? 1 : 0, s);
}

// FP64 rows -> NSL exact slices of BITS bits per element relative to 2^e, e = 1 +
// the binary exponent of the row's largest magnitude.  A warp per row, two
// consecutive elements per lane; bound by its writes (2 NSL bytes per element).
// 16 thousand rows of L = 320 into seven slices: 278 us with FP64 arithmetic.
template <int NSL, int BITS>
struct PackFixed64 {
  static __device__ __forceinline__ void run(const double *__restrict__ P, const int *__restrict__ list,
                                             const int *__restrict__ count, int nrows, int nsub, int stride, int L,
                                             int kp, uint16_t *__restrict__ A, int *__restrict__ rows_out,
                                             int *__restrict__ exps, long dst_stride, long dst_off,
                                             const int *__restrict__ scale, const uint3 bid,
                                             const uint3 gdim) {
    assume_global(P, A, rows_out, exps);
    const int rows = count ? *count : nrows;
    const int lane = threadIdx.x & 31;
    const long nw = (long)gdim.x * (blockDim.x >> 5);
    for (long m = (long)bid.x * (blockDim.x >> 5) + (threadIdx.x >> 5); m < rows; m += nw) {
      const long phys = list ? (long)list[m] : (m / nsub) * stride + (m % nsub);
      const double *src = P + phys * L;
      const int *sc = scale ? scale + (m / nsub) * L : nullptr;  // element k is taken times 2^-sc[k]
      int mx = kNoExponent;
      for (int k = lane; k < L; k += 32) mx = max(mx, element_exponent(src[k], sc ? -sc[k] : 0));
      const int e = exponent_of_max(__reduce_max_sync(0xffffffffu, mx));
      if (lane == 0) {
        // the row of the result: the source row, or (m / nsub) * dst_stride + dst_off + m % nsub
        rows_out[m] = dst_stride > 0 ? (int)((m / nsub) * dst_stride + dst_off + m % nsub) : (int)phys;
        exps[m] = e;
      }
      uint16_t *dst = A + m * NSL * (long)kp;
      for (int k = 2 * lane; k < kp; k += 64) {
        uint16_t t0[NSL], t1[NSL];
        cut_slices<NSL, BITS>(k < L ? src[k] : 0.0, sc && k < L ? e + sc[k] : e, t0);
        cut_slices<NSL, BITS>(k + 1 < L ? src[k + 1] : 0.0, sc && k + 1 < L ? e + sc[k + 1] : e, t1);
  #pragma unroll
        for (int t = 0; t < NSL; ++t)
          *reinterpret_cast<uint32_t *>(dst + t * kp + k) = t0[t] | (static_cast<uint32_t>(t1[t]) << 16);
      }
    }
}
};
template <int NSL, int BITS>
__global__ void __launch_bounds__(256) k_pack_fixed64(const double *__restrict__ P, const int *__restrict__ list,
                                                      const int *__restrict__ count, int nrows, int nsub, int stride,
                                                      int L, int kp, uint16_t *__restrict__ A,
                                                      int *__restrict__ rows_out, int *__restrict__ exps,
                                                      long dst_stride, long dst_off,
                                                      const int *__restrict__ scale) {
  PackFixed64<NSL, BITS>::run(P, list, count, nrows, nsub, stride, L, kp, A, rows_out, exps, dst_stride, dst_off,
                              scale, blockIdx, gridDim);
}

template <int NSL, int BITS>
static cudaError_t pack_fixed64(const double *P, const int *list, const int *count, int nrows, int nsub, int stride,
                                int L, int kp, uint16_t *A, int *rows_out, int *exps, int blocks, cudaStream_t st,
                                long dst_stride, long dst_off, const int *scale) {
  return launch_or_record<PackFixed64<NSL, BITS>, 256>(k_pack_fixed64<NSL, BITS>, dim3(blocks), dim3(256), 0, st, P,
                                                       list, count, nrows, nsub > 0 ? nsub : 1, stride, L, kp, A,
                                                       rows_out, exps, dst_stride, dst_off, scale);
}

cudaError_t launch_pack_fixed64(const double *P, const int *list, const int *count, int nrows, int nsub, int stride,
                                int L, int kp, int nsl, int bits, uint16_t *A, int *rows_out, int *exps,
                                int max_rows, cudaStream_t st, long dst_stride, long dst_off,
                                const int *scale) {
  if (max_rows <= 0) return cudaSuccess;
  if (scale && (list || nsub <= 0)) return cudaErrorInvalidValue;
  long blocks = (max_rows + 7) / 8;
  if (blocks > 152 * 16) blocks = 152 * 16;
  const int nb = (int)blocks;
  if (nsl == 6 && bits == 8)
    return pack_fixed64<6, 8>(P, list, count, nrows, nsub, stride, L, kp, A, rows_out, exps, nb, st, dst_stride, dst_off,
                              scale);
  if (nsl == 7 && bits == 8)
    return pack_fixed64<7, 8>(P, list, count, nrows, nsub, stride, L, kp, A, rows_out, exps, nb, st, dst_stride, dst_off,
                              scale);
  if (nsl == 8 && bits == 7)
    return pack_fixed64<8, 7>(P, list, count, nrows, nsub, stride, L, kp, A, rows_out, exps, nb, st, dst_stride, dst_off,
                              scale);
  return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// Columns of per-walker matrices as fixed-point operand rows (the operands of
// the kinetic M products, whose contraction runs over the rows of G~^{-1},
// Bt and A_up): for walker w < W and column c < C of X_w = X + w xw
// ([R][C] row-major), operand row m = w C + c holds X_w[0..R)[c] (zero from R
// to kp) relative to 2^e, e = 1 + the binary exponent of the column's largest
// magnitude, cut into nsl exact slices of `bits` bits (FP64 X: 8 or 7 bits, up
// to eight slices; two-float X + Xlo: 8 bits, the remainder carried exactly)
// as k_pack_fixed cuts a row.
// exps[m] = e; rows_out[m] = w dst_stride + dst_off + c when rows_out is given.
// One CTA per (walker, 32 columns): the column maxima first, then tiles of 64
// rows through shared memory, so that the reads (32 consecutive columns of a
// row) and the writes (64 consecutive entries of one slice of an operand row)
// are both coalesced.
// ---------------------------------------------------------------------------
template <bool kF64, int NSL, int BITS>
struct PackCols {
  static __device__ __forceinline__ void run(const double *__restrict__ X64, const float *__restrict__ X32,
                                             const float *__restrict__ Xlo, size_t xw, int R, int C, int kp,
                                             uint16_t *__restrict__ A, int *__restrict__ exps,
                                             int *__restrict__ rows_out, long dst_stride, long dst_off,
                                             const int *__restrict__ scale, int sign, const uint3 bid, const uint3 gdim) {
    assume_global(A, exps);
    if constexpr (kF64) assume_global(X64); else assume_global(X32);
    __shared__ double t64[kF64 ? 64 : 1][33];
    __shared__ float th[kF64 ? 1 : 64][33], tl[kF64 ? 1 : 64][33];
    __shared__ int cmax[8][32];
    __shared__ int cexp[32];
    const int tid = threadIdx.x, cl = tid & 31, jr = tid >> 5;
    const int w = bid.y, c0 = bid.x * 32;
    const int c = c0 + cl;
    const size_t base = (size_t)w * xw;
    // row j is taken times 2^(sign scale[j]) (FP64)
    const int *sc = kF64 && scale ? scale + (size_t)w * R : nullptr;
    // the columns' largest magnitudes, as integer bits (FP64: their exponents)
    int mx = kF64 ? kNoExponent : 0;
    if (c < C)
      for (int j = jr; j < R; j += 8) {
        int h;
        if constexpr (kF64)
          h = element_exponent(X64[base + (size_t)j * C + c], sc ? sign * sc[j] : 0);
        else
          h = __float_as_int(fmaxf(0.0f, fabsf(X32[base + (size_t)j * C + c])));  // (NaN: 0)
        mx = h > mx ? h : mx;
      }
    cmax[jr][cl] = mx;
    __syncthreads();
    if (jr == 0) {
      for (int q = 1; q < 8; ++q) mx = cmax[q][cl] > mx ? cmax[q][cl] : mx;
      int e;
      if constexpr (kF64) {
        e = exponent_of_max(mx);
      } else {
        const float m = __int_as_float(mx);
        e = m > 0.0f ? ilogbf(m) + 1 : 0;
      }
      cexp[cl] = e;
      if (c < C) {
        exps[(size_t)w * C + c] = e;
        if (rows_out) rows_out[(size_t)w * C + c] = (int)(w * dst_stride + dst_off + c);
      }
    }
    __syncthreads();
    for (int j0 = 0; j0 < kp; j0 += 64) {
      // tile [64 rows][32 columns], zero past R or C
  #pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int jj = jr + 8 * q, j = j0 + jj;
        const bool in = j < R && c < C;
        if constexpr (kF64) {
          t64[jj][cl] = in ? X64[base + (size_t)j * C + c] : 0.0;
        } else {
          th[jj][cl] = in ? X32[base + (size_t)j * C + c] : 0.0f;
          tl[jj][cl] = (in && Xlo) ? Xlo[base + (size_t)j * C + c] : 0.0f;
        }
      }
      __syncthreads();
      // warp jr writes columns jr, jr + 8, jr + 16, jr + 24; lane: rows 2 lane, 2 lane + 1
  #pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        const int col = jr + 8 * cc, cg = c0 + col;
        if (cg >= C) continue;
        const int e = cexp[col];
        uint16_t sl[2][NSL];
  #pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int jj = 2 * (tid & 31) + h;
          if constexpr (kF64) {
            cut_slices<NSL, BITS>(t64[jj][col], sc && j0 + jj < R ? e - sign * sc[j0 + jj] : e, sl[h]);
          } else {
            float x = ldexpf(th[jj][col], 7 - e), xl = ldexpf(tl[jj][col], 7 - e);
  #pragma unroll
            for (int t = 0; t < NSL; ++t) {
              const float q = rintf(x);
              sl[h][t] = __bfloat16_as_ushort(__float2bfloat16_rn(q));
              const fdw r = two_sum(__fsub_rn(x, q), xl);
              x = __fmul_rn(r.hi, 256.0f);
              xl = __fmul_rn(r.lo, 256.0f);
            }
          }
        }
        uint16_t *dst = A + ((size_t)w * C + cg) * NSL * (size_t)kp + j0 + 2 * (tid & 31);
  #pragma unroll
        for (int t = 0; t < NSL; ++t)
          *reinterpret_cast<uint32_t *>(dst + (size_t)t * kp) = sl[0][t] | (static_cast<uint32_t>(sl[1][t]) << 16);
      }
      __syncthreads();
    }
}
};
template <bool kF64, int NSL, int BITS>
__global__ void __launch_bounds__(256) k_pack_cols(const double *__restrict__ X64, const float *__restrict__ X32,
                                                   const float *__restrict__ Xlo, size_t xw, int R, int C, int kp,
                                                   uint16_t *__restrict__ A, int *__restrict__ exps,
                                                   int *__restrict__ rows_out, long dst_stride, long dst_off,
                                                   const int *__restrict__ scale, int sign) {
  PackCols<kF64, NSL, BITS>::run(X64, X32, Xlo, xw, R, C, kp, A, exps, rows_out, dst_stride, dst_off, scale, sign,
                                 blockIdx, gridDim);
}

template <bool kF64, int NSL, int BITS>
static cudaError_t pack_cols(const double *X64, const float *X32, const float *Xlo, size_t xw, int R, int C, int kp,
                             int W, uint16_t *A, int *exps, int *rows_out, long dst_stride, long dst_off,
                             cudaStream_t st, const int *scale, int sign) {
  return launch_or_record<PackCols<kF64, NSL, BITS>, 256>(k_pack_cols<kF64, NSL, BITS>, dim3((C + 31) / 32, W),
                                                          dim3(256), 0, st, X64, X32, Xlo, xw, R, C, kp, A, exps,
                                                          rows_out, dst_stride, dst_off, scale, sign);
}

cudaError_t launch_pack_cols(const double *X64, const float *X32, const float *Xlo, size_t xw, int R, int C, int kp,
                             int W, uint16_t *A, int *exps, int *rows_out, long dst_stride, long dst_off,
                             cudaStream_t st, int nsl, int bits, const int *scale, int sign) {
  if (W <= 0 || C <= 0) return cudaSuccess;
  if (kp % 64 != 0 || kp < R || (X64 == nullptr) == (X32 == nullptr) || (scale && !X64)) return cudaErrorInvalidValue;
  if (X32 && nsl == 6 && bits == 8)
    return pack_cols<false, 6, 8>(X64, X32, Xlo, xw, R, C, kp, W, A, exps, rows_out, dst_stride, dst_off, st, scale,
                               sign);
  if (X64 && nsl == 6 && bits == 8)
    return pack_cols<true, 6, 8>(X64, X32, Xlo, xw, R, C, kp, W, A, exps, rows_out, dst_stride, dst_off, st, scale,
                               sign);
  if (X64 && nsl == 7 && bits == 8)
    return pack_cols<true, 7, 8>(X64, X32, Xlo, xw, R, C, kp, W, A, exps, rows_out, dst_stride, dst_off, st, scale,
                               sign);
  if (X64 && nsl == 8 && bits == 7)
    return pack_cols<true, 8, 7>(X64, X32, Xlo, xw, R, C, kp, W, A, exps, rows_out, dst_stride, dst_off, st, scale,
                               sign);
  return cudaErrorInvalidValue;
}

cudaError_t setup_umma_attributes() {
  // the largest opt-in shared memory per block (227 KB on this part), so that
  // two or more stages of every slice fit (with K chunks of 32 or 16)
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  g_smem_optin = optin < 220 * 1024 ? 220 * 1024 : optin;
  return cudaFuncSetAttribute(k_umma_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, g_smem_optin);
}

}  // namespace jagp
