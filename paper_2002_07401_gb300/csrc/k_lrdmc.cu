// k_lrdmc.cu -- lattice-regularised diffusion Monte Carlo (Sec. "Lattice
// regularized Monte Carlo"), FP64 path, guiding function Psi_G = Psi_T,
// continuous time.
//
// Hop k = 6 i + 2 d + s moves electron i by +a (s = 0) or -a (s = 1) along
// axis d.  Its ratio Psi_G(x') / Psi_G(x) needs no determinant: the new row
// (up electron) or column (down electron) of G~ is linear in phi(r'), so the
// determinant ratio is phi(r') . M_i with the kinetic contraction vectors
// M_i = sum_j G~^{-1}[j][i] Bt_j (up) or sum_j G~^{-1}[i'][j] A_up_j (down)
// that the local energy of the current configuration has already formed;
// the Jastrow factor contributes exp(dJ1 + dJ2).  The fixed-node,
// importance-sampled Green's function leaves x for x'_k at the rate
// t_k = (rho_k > 0 ? rho_k : gamma |rho_k|) / (2 a^2), and weights the
// walker by exp(-(e_L(x) - e_ref) dt) while it stays (the regularised
// potential of Eq. lrdmc_potential makes the column sum of the fixed-node
// Hamiltonian the continuous local energy).
//
// A projection runs in rounds: every walker with time left takes one hop
// (or ends) per round, a warp deciding for each walker; then the moved
// electrons' orbital rows and their lambda products, and, on a compact copy
// of the moved walkers' state, a refresh of G~^{-1} and the local energy of
// the new configurations (jagp_api.cu) prepare the next round.  Decisions read the Philox4x32-10 stream (walker, generation, hop, 2).
#include <atomic>

#include "jagp_group.cuh"
#include "jagp_launch.h"

namespace jagp {

namespace {

constexpr int kRatioThreads = 128;

// 2^(j / 64) as double-words (its FP32 rounding and the remainder)
__device__ const float2 kExpTab[64] = {
    {0x1.0000000000000p+0f, 0x0.0p+0f}, {0x1.02c9a40000000p+0f, -0x1.887fa00000000p-28f},
    {0x1.059b0e0000000p+0f, -0x1.9d4f520000000p-25f}, {0x1.0874520000000p+0f, -0x1.e2990e0000000p-26f},
    {0x1.0b55860000000p+0f, 0x1.9f31220000000p-25f}, {0x1.0e3ec40000000p+0f, -0x1.a585cc0000000p-25f},
    {0x1.11301e0000000p+0f, -0x1.fdb4960000000p-25f}, {0x1.1429aa0000000p+0f, 0x1.d525bc0000000p-25f},
    {0x1.172b840000000p+0f, -0x1.c157420000000p-27f}, {0x1.1a35be0000000p+0f, 0x1.6df96e0000000p-25f},
    {0x1.1d48740000000p+0f, -0x1.d2e8ca0000000p-25f}, {0x1.2063b80000000p+0f, 0x1.0c519a0000000p-25f},
    {0x1.2387a60000000p+0f, 0x1.ceac480000000p-25f}, {0x1.26b4560000000p+0f, 0x1.789f380000000p-26f},
    {0x1.29e9e00000000p+0f, -0x1.5c04240000000p-25f}, {0x1.2d285a0000000p+0f, 0x1.b900c20000000p-26f},
    {0x1.306fe00000000p+0f, 0x1.4636e20000000p-25f}, {0x1.33c08c0000000p+0f, -0x1.b37d200000000p-25f},
    {0x1.371a740000000p+0f, -0x1.18aac60000000p-25f}, {0x1.3a7db40000000p+0f, -0x1.634c020000000p-25f},
    {0x1.3dea640000000p+0f, 0x1.8246840000000p-25f}, {0x1.4160a20000000p+0f, 0x1.f72e2a0000000p-28f},
    {0x1.44e0860000000p+0f, 0x1.8624b40000000p-30f}, {0x1.486a2c0000000p+0f, -0x1.47d8660000000p-25f},
    {0x1.4bfdae0000000p+0f, -0x1.593abc0000000p-25f}, {0x1.4f9b280000000p+0f, -0x1.2c5a6c0000000p-25f},
    {0x1.5342b60000000p+0f, -0x1.2c56100000000p-25f}, {0x1.56f4740000000p+0f, -0x1.295b040000000p-25f},
    {0x1.5ab07e0000000p+0f, -0x1.5bd5ec0000000p-27f}, {0x1.5e76f20000000p+0f, -0x1.4a5bd60000000p-25f},
    {0x1.6247ec0000000p+0f, -0x1.f8b5500000000p-25f}, {0x1.6623880000000p+0f, 0x1.2a91120000000p-27f},
    {0x1.6a09e60000000p+0f, 0x1.9fcef40000000p-26f}, {0x1.6dfb240000000p+0f, -0x1.cd72e80000000p-27f},
    {0x1.71f75e0000000p+0f, 0x1.1d8bee0000000p-25f}, {0x1.75feb60000000p+0f, -0x1.37b3060000000p-25f},
    {0x1.7a11480000000p+0f, -0x1.829fd00000000p-25f}, {0x1.7e2f340000000p+0f, -0x1.2616340000000p-25f},
    {0x1.82589a0000000p+0f, -0x1.accc7c0000000p-26f}, {0x1.868d9a0000000p+0f, -0x1.2edb440000000p-26f},
    {0x1.8ace540000000p+0f, 0x1.15506e0000000p-27f}, {0x1.8f1aea0000000p+0f, -0x1.baa2320000000p-26f},
    {0x1.93737c0000000p+0f, -0x1.e647440000000p-25f}, {0x1.97d82a0000000p+0f, -0x1.0d8d840000000p-31f},
    {0x1.9c49180000000p+0f, 0x1.51f8480000000p-27f}, {0x1.a0c6680000000p+0f, -0x1.2886a60000000p-26f},
    {0x1.a5503c0000000p+0f, -0x1.b83b540000000p-25f}, {0x1.a9e6b60000000p+0f, -0x1.50c0480000000p-25f},
    {0x1.ae89fa0000000p+0f, -0x1.a94b140000000p-26f}, {0x1.b33a2c0000000p+0f, -0x1.ec3a820000000p-26f},
    {0x1.b7f7700000000p+0f, -0x1.a094380000000p-25f}, {0x1.bcc1ea0000000p+0f, -0x1.f687c60000000p-25f},
    {0x1.c199be0000000p+0f, -0x1.3d56b20000000p-27f}, {0x1.c67f120000000p+0f, 0x1.cafa2a0000000p-25f},
    {0x1.cb720e0000000p+0f, -0x1.8837cc0000000p-27f}, {0x1.d072d40000000p+0f, 0x1.40f1300000000p-25f},
    {0x1.d5818e0000000p+0f, -0x1.822dbc0000000p-27f}, {0x1.da9e600000000p+0f, 0x1.ed99420000000p-27f},
    {0x1.dfc9740000000p+0f, -0x1.908c940000000p-25f}, {0x1.e502ee0000000p+0f, 0x1.e2cffe0000000p-26f},
    {0x1.ea4afa0000000p+0f, 0x1.52486c0000000p-27f}, {0x1.efa1be0000000p+0f, 0x1.cc2b440000000p-25f},
    {0x1.f507660000000p+0f, -0x1.246eb00000000p-26f}, {0x1.fa7c180000000p+0f, 0x1.9e90d80000000p-28f},
};

// e^x = m 2^k, |x| <= 170, by a table (Tang, ACM TOMS 15 (1989) 144): x = (64 k + j)
// ln2 / 64 + r, |r| <= ln2 / 128, ln2 / 64 in three parts (the first of 10 bits, so
// that its product and the first subtraction are exact), m = 2^(j/64) (1 + r +
// r^2/2 + ...) with r, r^2 and the table in double-word, r^3/6 .. r^6/720 in FP32;
// relative error below 2^-46.  The exponent stays apart, so that products and
// quotients of such numbers neither overflow nor underflow on the way.
struct ExpParts {
  fdw m;
  int k;
};
__device__ __forceinline__ ExpParts dw_exp_parts(fdw x, const float2 *__restrict__ tab) {
  const float k = rintf(__fmul_rn(x.hi, 92.33248138427734f));
  fdw r = two_sum(__fmaf_rn(-k, 0x1.628p-7f, x.hi), x.lo);
  r = dw_add(r, dw_neg(two_prod(k, 0x1.90bfbep-17f)));
  r = fast_two_sum(r.hi, __fmaf_rn(-k, 0x1.1cf79ap-42f, r.lo));
  const int ki = static_cast<int>(k);
  const float2 t = tab[ki & 63];
  const float h = __fmul_rn(r.hi, r.hi), hl = __fmaf_rn(2.0f * r.hi, r.lo, __fmaf_rn(r.hi, r.hi, -h));  // r^2
  float q = __fmaf_rn(r.hi, 1.0f / 720.0f, 1.0f / 120.0f);
  q = __fmaf_rn(q, r.hi, 1.0f / 24.0f);
  q = __fmaf_rn(q, r.hi, 1.0f / 6.0f);
  q = __fmul_rn(q, __fmul_rn(h, r.hi));
  const fdw e = fast_two_sum(r.hi, 0.5f * h);  // e^r - 1 = e.hi + low
  const float low = __fadd_rn(__fadd_rn(__fmaf_rn(0.5f, hl, r.lo), q), e.lo);
  const fdw te = two_prod(t.x, e.hi);
  const float tl = __fmaf_rn(t.x, low, __fmaf_rn(t.y, e.hi, te.lo));
  const fdw u = fast_two_sum(t.x, te.hi);
  return {fast_two_sum(u.hi, __fadd_rn(u.lo, __fadd_rn(t.y, tl))), ki >> 6};
}
// m 2^k, |m| below 2^20 or so; rounded once where the result is subnormal
__device__ __forceinline__ fdw dw_scale(fdw m, int k) {
  if (k >= -100) {
    const float sc = __int_as_float((127 + (k < 127 ? k : 127)) << 23);
    return {__fmul_rn(m.hi, sc), __fmul_rn(m.lo, sc)};
  }
  return {ldexpf(m.hi, k), ldexpf(m.lo, k)};
}
// e^x for x <= 0 (0 below -104)
__device__ __forceinline__ fdw dw_exp_tab(fdw x, const float2 *__restrict__ tab) {
  if (!(x.hi > -104.0f)) return {x.hi != x.hi ? x.hi : 0.0f, 0.0f};
  const ExpParts p = dw_exp_parts(x, tab);
  return dw_scale(p.m, p.k);
}

// v as a double-word without FP64 instructions (a conversion occupies the FP64
// pipe for 16 clocks per warp): the leading 24 bits truncated, the other 29 as
// an integer.  Magnitudes outside FP32's normal range: 0, or an infinity / NaN.
__device__ __forceinline__ fdw dw_of_bits(double v) {
  const unsigned hi = static_cast<unsigned>(__double2hiint(v)), lo = static_cast<unsigned>(__double2loint(v));
  const unsigned sign = hi & 0x80000000u;
  const int e = static_cast<int>((hi >> 20) & 0x7ffu) - 1023;
  if (e > 127) {
    const bool nan = e == 1024 && ((hi & 0xfffffu) | lo) != 0u;
    return {__uint_as_float(sign | (nan ? 0x7fc00000u : 0x7f800000u)), 0.0f};
  }
  if (e < -126) return {0.0f, 0.0f};
  const unsigned scale = sign | static_cast<unsigned>(e + 127) << 23;  // +-2^e
  const float h = __uint_as_float(scale | (hi & 0xfffffu) << 3 | lo >> 29);
  const float l = __fmul_rn(__fmul_rn(static_cast<float>(static_cast<int>(lo & 0x1fffffffu)), 0x1p-52f),
                            __uint_as_float(scale));
  return fast_two_sum(h, l);
}

// warp-wide double-word sum; dw_add is commutative, so every lane of the
// butterfly ends with the same value
__device__ __forceinline__ fdw warp_sum_dw(fdw v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const fdw u{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
    v = dw_add(v, u);
  }
  return v;
}

// Squared distances r'^2 of the six hops from a centre at displacement d of the
// electron, r^2 + a^2 +- 2 a d_q.  This cancels where a hop lands near the centre
// (near: r'^2 below a quarter of r^2 + a^2): such centres are left to hop_from.
struct HopDist {
  fdw base;     // r^2 + a^2
  fdw step[3];  // 2 a d_q
  __device__ __forceinline__ fdw r2(int k) const {
    return dw_add(base, (k & 1) ? dw_neg(step[k >> 1]) : step[k >> 1]);
  }
  // the smallest r'^2, to FP32
  __device__ __forceinline__ float least() const {
    return base.hi - fmaxf(fmaxf(fabsf(step[0].hi), fabsf(step[1].hi)), fabsf(step[2].hi));
  }
  __device__ __forceinline__ bool near() const { return least() < 0.25f * base.hi; }
  // near a shell's atom the distance itself (a Slater shell), the exponents of a quotient of
  // Gaussians (an error of zeta (r^2 + a^2) units) and, closer, the polynomials lose bits
  __device__ __forceinline__ bool near_shell(int rad, float zeta) const {
    const float l = least();
    return l < 0.015625f * base.hi || (l < 0.25f * base.hi && (rad || zeta * base.hi > 4.0f));
  }
};
__device__ __forceinline__ HopDist hop_dist(const DwDisp &d, fdw two_a, fdw a2) {
  return {dw_add(d.r2, a2), {dw_mul(two_a, d.x), dw_mul(two_a, d.y), dw_mul(two_a, d.z)}};
}
// the displacement after hop k, its square a sum of three squares
__device__ __forceinline__ DwDisp hop_from(const DwDisp &d, fdw a, int k) {
  const fdw s = (k & 1) ? dw_neg(a) : a;
  DwDisp h = d;
  if (k < 2) h.x = dw_add(d.x, s);
  else if (k < 4) h.y = dw_add(d.y, s);
  else h.z = dw_add(d.z, s);
  h.r2 = dw_add(dw_add(dw_mul(h.x, h.x), dw_mul(h.y, h.y)), dw_mul(h.z, h.z));
  return h;
}
__device__ __forceinline__ DwDisp dw_between(const fdw *p, const fdw *q) {
  DwDisp d;
  d.x = dw_add(p[0], dw_neg(q[0]));
  d.y = dw_add(p[1], dw_neg(q[1]));
  d.z = dw_add(p[2], dw_neg(q[2]));
  d.r2 = dw_add(dw_add(dw_mul(d.x, d.x), dw_mul(d.y, d.y)), dw_mul(d.z, d.z));
  return d;
}

// one-body term of one atom, -c^3 u(c r), u(s) = (1 - e^{-b s}) / (2b) (s / 2 at b = 0)
__device__ __forceinline__ fdw j1_term_dw(fdw c, fdw mc3, fdw b, fdw inv2b, bool b0, fdw r,
                                          const float2 *__restrict__ tab) {
  const fdw sc = dw_mul(c, r);
  const fdw u =
      b0 ? dw_mul_f(sc, 0.5f) : dw_mul(dw_add_f(dw_neg(dw_exp_tab(dw_neg(dw_mul(b, sc)), tab)), 1.0f), inv2b);
  return dw_mul(mc3, u);
}

// pair term r / (k (1 + b r)), 1/k = kinv (a power of two)
__device__ __forceinline__ fdw j2_term_dw(fdw b, float kinv, fdw r) {
  return dw_mul_f(dw_mul(r, dw_recip(dw_add_f(dw_mul(b, r), 1.0f))), kinv);
}

// rho[w][k] for every hop of every walker still active: one CTA per walker, a
// warp per electron and its six hops (lanes over shells, atoms and electrons),
// in double-word FP32 arithmetic (relative error a few units of 2^-46).  Bound by
// its FP32 instructions, so that what the six hops share is formed once: a hop by
// +-a along q changes r^2 by a^2 +- 2 a d_q, so a Gaussian's six radial factors are
// e^{-zeta (r^2 + a^2)} times or over e^{-2 zeta a d_q} (four exponentials, not
// six), and sum_c M_c P_c, a polynomial of degree two at most, follows from its
// value, gradient and second derivatives at the electron.  Where a hop lands near a
// centre these cancel: the few shells, atoms and electrons it concerns are passed by
// and taken afterwards, hop by hop from the hop's own displacement (in the same
// loops that code took the kernel from 72 to 96 registers, and a generation from 36.4 to
// 39.5 ms).  Conversions are done with integer instructions.  A generation of 1024
// walkers of 16 He, 26 rounds: 22.0 -> 10.2 ms against six separate evaluations.
// ATOMS: the atoms' double-words in shared memory too (some five thousand do not fit).
template <bool ATOMS>
__global__ void __launch_bounds__(kRatioThreads, 7) k_lrdmc_ratios(DevSystem s, const double *__restrict__ r,
                                                                    const double *__restrict__ mbuf,
                                                                    const int *__restrict__ active, double a,
                                                                    double *__restrict__ rho) {
  extern __shared__ fdw xd[];         // the walker's positions [N][3], then per atom R, c, -c^3
  __shared__ float2 tab[64];
  const int w = blockIdx.x, N = s.N, L = s.L, na = s.n_atoms;
  fdw *const ad = xd + 3 * N;
  if (!active[w]) return;
  for (int t = threadIdx.x; t < 3 * N; t += kRatioThreads) xd[t] = dw_of_bits(r[(size_t)w * N * 3 + t]);
  // atom t: R, c, -c^3
  auto split_atom = [&](int t, fdw *q) {
    for (int k = 0; k < 3; ++k) q[k] = dw_of_bits(s.R[3 * t + k]);
    const double c = s.c1[t];
    q[3] = dw_of_bits(c);
    q[4] = dw_of_bits(-c * c * c);
  };
  if constexpr (ATOMS)
    for (int t = threadIdx.x; t < na; t += kRatioThreads) split_atom(t, ad + 5 * t);
  // atom t's five numbers, in shared memory or in q
  auto atom = [&](int t, fdw *q) -> const fdw * {
    if constexpr (ATOMS) return ad + 5 * t;
    split_atom(t, q);
    return q;
  };
  for (int t = threadIdx.x; t < 64; t += kRatioThreads) tab[t] = kExpTab[t];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool b0 = s.b_ea == 0.0;
  const fdw bea = dw_of_bits(s.b_ea), inv2b = dw_of_bits(b0 ? 0.0 : 0.5 / s.b_ea);
  const fdw ah = dw_of_bits(a), a2 = dw_mul(ah, ah), two_a{2.0f * ah.hi, 2.0f * ah.lo};
  // pair constants [same spin, opposite]
  double k2[2], bb2[2];
  j2_params(s, true, &k2[0], &bb2[0]);
  j2_params(s, false, &k2[1], &bb2[1]);
  const fdw b2[2] = {dw_of_bits(bb2[0]), dw_of_bits(bb2[1])};
  const float kinv2[2] = {k2[0] == 4.0 ? 0.25f : 0.5f, k2[1] == 4.0 ? 0.25f : 0.5f};
  for (int i = warp; i < N; i += kRatioThreads / 32) {
    const fdw *od = xd + 3 * i;
    fdw dot[6], dj[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) dot[k] = dj[k] = fdw{0.0f, 0.0f};
    const double *Mi = mbuf + ((size_t)w * N + i) * L;
    unsigned later = 0;  // what has a hop near: bit 0 a shell, 1 an atom, 2 an electron
    for (int sh = lane; sh < s.n_shells; sh += 32) {
      const float4 gh = s.shell_dw[2 * sh], gl = s.shell_dw[2 * sh + 1];
      const int info = s.shell_info[sh], off = shell_off(info), l = shell_l(info), rad = shell_rad(info);
      const fdw zeta{gh.w, gl.w};
      const fdw at[3] = {{gh.x, gl.x}, {gh.y, gl.y}, {gh.z, gl.z}};
      const DwDisp d = displacement(od, at);
      // every hop's value is 0 in FP32 (e^-104) where even the nearest one is that far
      const float far = fmaxf(fmaxf(fabsf(d.x.hi), fabsf(d.y.hi)), fabsf(d.z.hi));
      const float near2 = fmaxf(d.r2.hi + a2.hi - 2.0f * ah.hi * far, 0.0f);
      if (gh.w * (rad ? sqrtf(near2) : near2) > 105.0f) continue;
      const HopDist h = hop_dist(d, two_a, a2);
      if (h.near_shell(rad, gh.w)) {
        later |= 1u;
        continue;
      }
      // S = sum_c M_c P_c at the electron, its gradient and half its second derivatives
      const fdw m0 = dw_of_bits(Mi[off]);
      fdw S0, Sq[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, Cq[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
      if (l == 0) {
        S0 = m0;
      } else if (l == 1) {
        Sq[0] = m0;
        Sq[1] = dw_of_bits(Mi[off + 1]);
        Sq[2] = dw_of_bits(Mi[off + 2]);
        S0 = dw_add(dw_add(dw_mul(Sq[0], d.x), dw_mul(Sq[1], d.y)), dw_mul(Sq[2], d.z));
      } else {
        const fdw m1 = dw_of_bits(Mi[off + 1]), m2 = dw_of_bits(Mi[off + 2]), m3 = dw_of_bits(Mi[off + 3]),
                  m4 = dw_of_bits(Mi[off + 4]);
        // P = xy, yz, zx, x^2 - y^2, 2 z^2 - x^2 - y^2: S = x (S_x / 2) + y (S_y / 2) + z (S_z / 2)
        Cq[0] = dw_add(m3, dw_neg(m4));
        Cq[1] = dw_neg(dw_add(m3, m4));
        Cq[2] = fdw{2.0f * m4.hi, 2.0f * m4.lo};
        const fdw x2{2.0f * d.x.hi, 2.0f * d.x.lo}, y2{2.0f * d.y.hi, 2.0f * d.y.lo}, z2{2.0f * d.z.hi, 2.0f * d.z.lo};
        Sq[0] = dw_add(dw_add(dw_mul(m0, d.y), dw_mul(m2, d.z)), dw_mul(Cq[0], x2));
        Sq[1] = dw_add(dw_add(dw_mul(m0, d.x), dw_mul(m1, d.z)), dw_mul(Cq[1], y2));
        Sq[2] = dw_add(dw_add(dw_mul(m1, d.y), dw_mul(m2, d.x)), dw_mul(Cq[2], z2));
        const fdw t = dw_add(dw_add(dw_mul(Sq[0], d.x), dw_mul(Sq[1], d.y)), dw_mul(Sq[2], d.z));
        S0 = fdw{0.5f * t.hi, 0.5f * t.lo};
      }
      // the six hops' S: S0 +- a S_q + a^2 C_q
      fdw S[6];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        if (l == 0) {
          S[2 * q] = S[2 * q + 1] = S0;
        } else {
          const fdw c = l == 2 ? dw_add(S0, dw_mul(a2, Cq[q])) : S0, g = dw_mul(ah, Sq[q]);
          S[2 * q] = dw_add(c, g);
          S[2 * q + 1] = dw_add(c, dw_neg(g));
        }
      }
      if (rad || gh.w * h.base.hi > 168.0f) {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const fdw r2 = h.r2(k);
          dot[k] = dw_add(dot[k], dw_mul(dw_exp_tab(dw_neg(dw_mul(zeta, rad ? dw_sqrt(r2) : r2)), tab), S[k]));
        }
      } else {
        // zeta (r^2 + a^2) <= 168 bounds 2 zeta a |d_q| too
        const ExpParts e0 = dw_exp_parts(dw_neg(dw_mul(zeta, h.base)), tab);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const ExpParts f = dw_exp_parts(dw_neg(dw_mul(zeta, h.step[q])), tab);
          dot[2 * q] = dw_add(dot[2 * q], dw_mul(dw_scale(dw_mul(e0.m, f.m), e0.k + f.k), S[2 * q]));
          dot[2 * q + 1] =
              dw_add(dot[2 * q + 1], dw_mul(dw_scale(dw_mul(e0.m, dw_recip(f.m)), e0.k - f.k), S[2 * q + 1]));
        }
      }
    }
    if (s.use_j1) {
      for (int at = lane; at < na; at += 32) {
        fdw buf[5];
        const fdw *R = atom(at, buf), cd = R[3], mc3 = R[4];
        const DwDisp d = dw_between(od, R);
        const HopDist h = hop_dist(d, two_a, a2);
        if (h.near()) {
          later |= 2u;
          continue;
        }
        const fdw f0 = j1_term_dw(cd, mc3, bea, inv2b, b0, dw_sqrt(d.r2), tab);
#pragma unroll
        for (int k = 0; k < 6; ++k)
          dj[k] = dw_add(dj[k], dw_add(j1_term_dw(cd, mc3, bea, inv2b, b0, dw_sqrt(h.r2(k)), tab), dw_neg(f0)));
      }
    }
    if (s.use_j2) {
      const bool up = i < s.n_up;
      for (int q = lane; q < N; q += 32) {
        if (q == i) continue;
        const int o = (q < s.n_up) == up ? 0 : 1;
        const fdw b = o ? b2[1] : b2[0];
        const float kinv = o ? kinv2[1] : kinv2[0];
        const DwDisp d = dw_between(od, xd + 3 * q);
        const HopDist h = hop_dist(d, two_a, a2);
        if (h.near()) {
          later |= 4u;
          continue;
        }
        const fdw f0 = j2_term_dw(b, kinv, dw_sqrt(d.r2));
#pragma unroll
        for (int k = 0; k < 6; ++k)
          dj[k] = dw_add(dj[k], dw_add(j2_term_dw(b, kinv, dw_sqrt(h.r2(k))), dw_neg(f0)));
      }
    }
    // lane k < 6 has hop k's sums
    fdw hd{0.0f, 0.0f}, hj{0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const fdw dk = warp_sum_dw(dot[k]), jk = warp_sum_dw(dj[k]);
      if (lane == k) {
        hd = dk;
        hj = jk;
      }
    }
    later = __reduce_or_sync(0xffffffffu, later);
    if (later & 1u)
      for (int t0 = 0; t0 < s.n_shells; t0 += 32) {
        auto from = [&](int sh) {
          const float4 gh = s.shell_dw[2 * sh], gl = s.shell_dw[2 * sh + 1];
          const fdw at[3] = {{gh.x, gl.x}, {gh.y, gl.y}, {gh.z, gl.z}};
          return displacement(od, at);
        };
        const int mine = t0 + lane;
        unsigned left = __ballot_sync(
            0xffffffffu, mine < s.n_shells && hop_dist(from(mine), two_a, a2)
                                                  .near_shell(shell_rad(s.shell_info[mine]), s.shell_dw[2 * mine].w));
        for (; left; left &= left - 1u) {
          const int sh = t0 + __ffs(left) - 1, info = s.shell_info[sh];
          const double *Ms = Mi + shell_off(info);
          const int l = shell_l(info), rad = shell_rad(info);
          const DwDisp h = hop_from(from(sh), ah, lane);
          fdw S = dw_of_bits(Ms[0]);
          if (l > 0) {
            S = dw_mul(S, l == 1 ? h.x : dw_mul(h.x, h.y));
            S = dw_add(S, dw_mul(dw_of_bits(Ms[1]), l == 1 ? h.y : dw_mul(h.y, h.z)));
            S = dw_add(S, dw_mul(dw_of_bits(Ms[2]), l == 1 ? h.z : dw_mul(h.z, h.x)));
          }
          if (l > 1) {
            S = dw_add(S, dw_mul(dw_of_bits(Ms[3]), dw_add(dw_mul(h.x, h.x), dw_neg(dw_mul(h.y, h.y)))));
            S = dw_add(S, dw_mul(dw_of_bits(Ms[4]), dw_add(dw_mul_f(dw_mul(h.z, h.z), 3.0f), dw_neg(h.r2))));
          }
          const fdw x = dw_mul(fdw{s.shell_dw[2 * sh].w, s.shell_dw[2 * sh + 1].w}, rad ? dw_sqrt(h.r2) : h.r2);
          hd = dw_add(hd, dw_mul(S, dw_exp_tab(dw_neg(x), tab)));
        }
      }
    if (later & 2u)
      for (int t0 = 0; t0 < na; t0 += 32) {
        fdw buf[5];
        const int mine = t0 + lane;
        unsigned left = __ballot_sync(
            0xffffffffu, mine < na && hop_dist(dw_between(od, atom(mine, buf)), two_a, a2).near());
        for (; left; left &= left - 1u) {
          const fdw *R = atom(t0 + __ffs(left) - 1, buf);
          const DwDisp d = dw_between(od, R);
          const fdw f0 = j1_term_dw(R[3], R[4], bea, inv2b, b0, dw_sqrt(d.r2), tab);
          hj = dw_add(hj, dw_add(j1_term_dw(R[3], R[4], bea, inv2b, b0, dw_sqrt(hop_from(d, ah, lane).r2), tab),
                                 dw_neg(f0)));
        }
      }
    if (later & 4u)
      for (int t0 = 0; t0 < N; t0 += 32) {
        const int mine = t0 + lane;
        unsigned left = __ballot_sync(0xffffffffu, mine < N && mine != i &&
                                                       hop_dist(dw_between(od, xd + 3 * mine), two_a, a2).near());
        for (; left; left &= left - 1u) {
          const int q = t0 + __ffs(left) - 1, o = (q < s.n_up) == (i < s.n_up) ? 0 : 1;
          const fdw b = o ? b2[1] : b2[0];
          const float kinv = o ? kinv2[1] : kinv2[0];
          const DwDisp d = dw_between(od, xd + 3 * q);
          hj = dw_add(hj, dw_add(j2_term_dw(b, kinv, dw_sqrt(hop_from(d, ah, lane).r2)),
                                 dw_neg(j2_term_dw(b, kinv, dw_sqrt(d.r2)))));
        }
      }
    if (lane < 6)
      rho[(size_t)w * 6 * N + 6 * i + lane] = (static_cast<double>(hd.hi) + static_cast<double>(hd.lo)) *
                                              exp(static_cast<double>(hj.hi) + static_cast<double>(hj.lo));
  }
}

// Start of a projection: time left tau, log-weight 0, no hops; walkers whose
// G~ is singular (or positions non-finite) do not take part (flag 2).
__global__ void k_lrdmc_start(const int *__restrict__ status, int W, double tau, double *__restrict__ left,
                              double *__restrict__ lw, int *__restrict__ hops, int *__restrict__ flags,
                              int *__restrict__ active) {
  const int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= W) return;
  const bool bad = (status[w] & (JAGP_WS_SINGULAR | JAGP_WS_NONFINITE)) != 0;
  left[w] = tau;
  lw[w] = 0.0;
  hops[w] = 0;
  flags[w] = bad ? 2 : 0;
  active[w] = bad ? 0 : 1;
}

// One round's decision per walker, a warp each: the rates and Gamma from rho, the
// wait tau_xi = -ln(1 - xi) / Gamma; the walker ends (log-weight less the time
// left times e_L - e_ref) or hops to the first k in hop order whose running rate
// sum exceeds u Gamma (a non-finite Gamma or e_L ends the walker with flag 4).
// A lane takes consecutive hops and the running sums come from a warp scan: one
// thread adding 12 N rates one after another took 86 us a round at N = 32, this 13.  A moved electron's row goes to the up or down list (w n_up + row)
// for the lambda products, the walker to list_w; cnt[2] counts the walkers
// that moved (those still active).
__global__ void __launch_bounds__(128) k_lrdmc_decide(
    DevSystem s, double *__restrict__ r, const double *__restrict__ rho, const double *__restrict__ eL,
    const int *__restrict__ status, int W, uint32_t walker0, uint32_t gen, double a, double gamma, double e_ref,
    int max_hops, double *__restrict__ left, double *__restrict__ lw, int *__restrict__ hops, int *__restrict__ flags,
    int *__restrict__ active, int *__restrict__ moved, int *__restrict__ list_up, int *__restrict__ list_dn,
    int *__restrict__ list_w, int *__restrict__ cnt) {
  const int w = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)), lane = threadIdx.x & 31;
  if (w >= W) return;
  const bool first = lane == 0;
  if (first) moved[w] = -1;
  if (!active[w]) return;
  if (status[w] & (JAGP_WS_SINGULAR | JAGP_WS_NONFINITE)) {
    if (first) {
      flags[w] |= 2;
      active[w] = 0;
    }
    return;
  }
  const int N = s.N, n = s.n_up, K = 6 * N, per = (K + 31) / 32, k0 = lane * per, k1 = min(K, k0 + per);
  const double *q = rho + (size_t)w * K;
  const double c = 1.0 / (2.0 * a * a);
  double mine = 0.0;
  for (int k = k0; k < k1; ++k) mine += (q[k] > 0.0 ? q[k] : -gamma * q[k]) * c;
  double incl = mine;  // sums up to and with this lane's hops
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const double before = __shfl_up_sync(0xffffffffu, incl, 1), G = __shfl_sync(0xffffffffu, incl, 31);
  const double e = eL[w];
  if (!isfinite(G) || !isfinite(e)) {
    if (first) {
      flags[w] |= 4;
      active[w] = 0;
    }
    return;
  }
  const int h = hops[w];
  const double time = left[w];
  if (h >= max_hops) {
    if (first) {
      flags[w] |= 1;
      lw[w] -= time * (e - e_ref);
      active[w] = 0;
    }
    return;
  }
  uint32_t o[4] = {walker0 + (uint32_t)w, gen, (uint32_t)h, 2u};
  philox4x32_10(o, s.key0, s.key1);
  const double xi = ((double)o[0] + 0.5) * 0x1p-32;
  const double wait = G > 0.0 ? -log(1.0 - xi) / G : INFINITY;
  if (wait >= time) {
    if (first) {
      lw[w] -= time * (e - e_ref);
      active[w] = 0;
    }
    return;
  }
  // the first hop whose running sum exceeds thr, else the last one with a rate
  const double thr = ((double)o[1] + 0.5) * 0x1p-32 * G;
  double run = lane ? before : 0.0;
  int hit = K, last = -1;
  for (int k = k0; k < k1 && hit == K; ++k) {
    const double t = (q[k] > 0.0 ? q[k] : -gamma * q[k]) * c;
    run += t;
    if (t > 0.0) {
      last = k;
      if (run > thr) hit = k;
    }
  }
  hit = static_cast<int>(__reduce_min_sync(0xffffffffu, static_cast<unsigned>(hit)));
  last = __reduce_max_sync(0xffffffffu, last);
  if (!first) return;
  const int k = hit < K ? hit : last;
  lw[w] -= wait * (e - e_ref);
  left[w] = time - wait;
  const int i = k / 6, d = (k % 6) / 2;
  double *x = r + ((size_t)w * N + i) * 3 + d;
  *x = (k & 1) ? *x - a : *x + a;
  hops[w] = h + 1;
  moved[w] = i;
  if (i < n)
    list_up[atomicAdd(cnt, 1)] = w * n + i;
  else
    list_dn[atomicAdd(cnt + 1, 1)] = w * n + (i - n);
  list_w[atomicAdd(cnt + 2, 1)] = w;
}

// Per-walker arrays between the state and the compact state of this round's
// moved walkers: gather dst[j] = src[list[j]], scatter dst[list[j]] = src[j],
// in 16-byte words where size and addresses allow, else 4-byte words (every
// per-walker size is a multiple of 4 bytes).  Bound by memory: a CTA per walker and
// array, four words in flight per thread (one CTA for all arrays of a walker and
// 4-byte words took 52 us per copy in a generation of 1024 walkers of 16 He, now 17).
template <typename V>
__device__ __forceinline__ void copy_words(V *__restrict__ d, const V *__restrict__ s, size_t words) {
  for (size_t t0 = threadIdx.x; t0 < words; t0 += 4 * (size_t)blockDim.x) {
    V v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (t0 + (size_t)q * blockDim.x < words) v[q] = s[t0 + (size_t)q * blockDim.x];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (t0 + (size_t)q * blockDim.x < words) d[t0 + (size_t)q * blockDim.x] = v[q];
  }
}
__global__ void __launch_bounds__(256) k_walker_copy(WalkerCopies cp, const int *__restrict__ list, int scatter) {
  const int j = blockIdx.x, w = list[j], a = blockIdx.y;
  const size_t bytes = cp.c[a].bytes;
  const char *s = reinterpret_cast<const char *>(cp.c[a].src) + (size_t)(scatter ? j : w) * bytes;
  char *d = reinterpret_cast<char *>(cp.c[a].dst) + (size_t)(scatter ? w : j) * bytes;
  if ((bytes | reinterpret_cast<size_t>(s) | reinterpret_cast<size_t>(d)) % 16 == 0)
    copy_words(reinterpret_cast<uint4 *>(d), reinterpret_cast<const uint4 *>(s), bytes / 16);
  else
    copy_words(reinterpret_cast<uint32_t *>(d), reinterpret_cast<const uint32_t *>(s), bytes / 4);
}

// Orbital values of each moved electron at its new position into the
// proposal table (row w n_up + row of its spin) and, for an up electron, into
// the current table phi_up.
__global__ void __launch_bounds__(128) k_lrdmc_rows(DevSystem s, const double *__restrict__ r,
                                                     const int *__restrict__ moved, double *__restrict__ pprop,
                                                     double *__restrict__ phi_up) {
  const int w = blockIdx.x, i = moved[w];
  if (i < 0) return;
  const int n = s.n_up, L = s.L;
  const double *p = r + ((size_t)w * s.N + i) * 3;
  const bool up = i < n;
  const size_t row = (size_t)w * n + (up ? i : i - n);
  for (int sh = threadIdx.x; sh < s.n_shells; sh += blockDim.x) {
    const double4 g = s.shell_geo[sh];
    const int info = s.shell_info[sh], off = shell_off(info);
    double v[5];
    const int nc = shell_values(info, g.w, p[0] - g.x, p[1] - g.y, p[2] - g.z, v);
    for (int c = 0; c < nc; ++c) {
      pprop[row * L + off + c] = v[c];
      if (up) phi_up[row * L + off + c] = v[c];
    }
  }
}

// End of a projection: weight *= exp(log-weight), e_L of the final configuration.
__global__ void k_lrdmc_finish(int W, const double *__restrict__ lw, const double *__restrict__ eL_cur,
                               double *__restrict__ weight, double *__restrict__ eL_out) {
  const int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= W) return;
  weight[w] *= exp(lw[w]);
  if (eL_out) eL_out[w] = eL_cur[w];
}

// Reconfiguration (Eqs. branching-1, branching-2) by systematic resampling, one
// CTA: z from Philox (0, g, 0, 3); new walker j takes the first old walker whose
// running weight sum exceeds (j + z) S / W; stats = (wbar, ebar).  Weights reset
// to 1.  Threads take consecutive walkers and scan their sums (run [W], scratch);
// one thread alone took 0.67 ms at W = 1024.
constexpr int kSelectThreads = 1024;
__global__ void __launch_bounds__(kSelectThreads) k_lrdmc_select(int W, uint32_t gen, uint32_t key0, uint32_t key1,
                                                                 double *__restrict__ weight,
                                                                 const double *__restrict__ eL,
                                                                 double *__restrict__ run, int *__restrict__ parent,
                                                                 double *__restrict__ stats) {
  __shared__ double ws[32], we[32];
  __shared__ int wl[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = (W + kSelectThreads - 1) / kSelectThreads, b0 = min(W, tid * per), b1 = min(W, b0 + per);
  double sum = 0.0, se = 0.0;
  int last = 0;  // the last walker with a weight
  for (int b = b0; b < b1; ++b) {
    sum += weight[b];
    se += weight[b] * eL[b];
    if (weight[b] > 0.0) last = b;
  }
  double incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  se = warp_sum(se);
  last = __reduce_max_sync(0xffffffffu, last);
  if (lane == 31) ws[warp] = incl;
  if (lane == 0) {
    we[warp] = se;
    wl[warp] = last;
  }
  __syncthreads();
  double base = 0.0, S = 0.0, Se = 0.0;
  last = 0;
  for (int q = 0; q < kSelectThreads / 32; ++q) {
    if (q < warp) base += ws[q];
    S += ws[q];
    Se += we[q];
    last = max(last, wl[q]);
  }
  const double before = __shfl_up_sync(0xffffffffu, incl, 1);
  double acc = lane ? base + before : base;
  for (int b = b0; b < b1; ++b) {
    acc += weight[b];
    run[b] = acc;
  }
  uint32_t o[4] = {0u, gen, 0u, 3u};
  philox4x32_10(o, key0, key1);
  const double z = ((double)o[0] + 0.5) * 0x1p-32;
  __syncthreads();  // run[] complete (one CTA: its own writes)
  for (int j = tid; j < W; j += kSelectThreads) {
    const double thr = ((double)j + z) * S / W;
    int lo = 0, hi = W;  // the first b with run[b] > thr
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (run[mid] > thr)
        hi = mid;
      else
        lo = mid + 1;
    }
    // (where two threads' walkers meet, the running sum is within rounding only: a
    // walker without weight gives way to the next one that has some)
    while (lo < W && !(weight[lo] > 0.0)) ++lo;
    parent[j] = lo < W ? lo : last;
  }
  __syncthreads();  // (every weight has been read)
  for (int j = tid; j < W; j += kSelectThreads) weight[j] = 1.0;
  if (tid == 0) {
    stats[0] = S / W;
    stats[1] = Se / S;
  }
}

// r_new[j] = r_old[parent[j]] (positions of the new population)
__global__ void k_lrdmc_gather(const double *__restrict__ r_old, const int *__restrict__ parent, int W, int N3,
                               double *__restrict__ r_new) {
  const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long)W * N3) return;
  const int j = (int)(t / N3), c = (int)(t % N3);
  r_new[t] = r_old[(size_t)parent[j] * N3 + c];
}

// E = sum_{n >= p} G_n ebar_n / sum G_n, G_n = prod_{j=1..p} wbar_{n-j}, as
// exponentials of log sums less their largest (one thread, in order)
__global__ void k_lrdmc_energy(const double *__restrict__ wbar, const double *__restrict__ ebar, int T, int p,
                               double *__restrict__ E) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double mx = -INFINITY;
  for (int n = p; n < T; ++n) {
    double l = 0.0;
    for (int j = 1; j <= p; ++j) l += log(wbar[n - j]);
    mx = fmax(mx, l);
  }
  double num = 0.0, den = 0.0;
  for (int n = p; n < T; ++n) {
    double l = 0.0;
    for (int j = 1; j <= p; ++j) l += log(wbar[n - j]);
    const double g = exp(l - mx);
    num += g * ebar[n];
    den += g;
  }
  E[0] = num / den;
}

}  // namespace

cudaError_t launch_lrdmc_ratios(const DevSystem &s, const double *r, const double *mbuf, const int *active, double a,
                                double *rho, int W, cudaStream_t st) {
  if (W <= 0) return cudaSuccess;
  const size_t pos = (size_t)s.N * 3 * sizeof(fdw), smem = pos + (size_t)s.n_atoms * 5 * sizeof(fdw);
  if (smem > 200 * 1024) {
    k_lrdmc_ratios<false><<<W, kRatioThreads, pos, st>>>(s, r, mbuf, active, a, rho);  // (N <= 1024: 24 KB)
    return cudaGetLastError();
  }
  if (smem > kRaiseSmem) {  // (static shared memory comes on top)
    static std::atomic<unsigned char> raised[64];
    const cudaError_t e = group_raise_smem(reinterpret_cast<const void *>(k_lrdmc_ratios<true>), raised);
    if (e != cudaSuccess) return e;
  }
  k_lrdmc_ratios<true><<<W, kRatioThreads, smem, st>>>(s, r, mbuf, active, a, rho);
  return cudaGetLastError();
}

cudaError_t launch_lrdmc_start(const int *status, int W, double tau, LrdmcWork &lw, cudaStream_t st) {
  if (W <= 0) return cudaSuccess;
  k_lrdmc_start<<<(W + 127) / 128, 128, 0, st>>>(status, W, tau, lw.left, lw.lw, lw.hops, lw.flags, lw.active);
  return cudaGetLastError();
}

cudaError_t launch_lrdmc_decide(const DevSystem &s, double *r, const double *eL, const int *status, int W,
                                uint32_t walker0, uint32_t gen, double a, double gamma, double e_ref, int max_hops,
                                LrdmcWork &lw, cudaStream_t st) {
  if (W <= 0) return cudaSuccess;
  k_lrdmc_decide<<<(W + 3) / 4, 128, 0, st>>>(s, r, lw.rho, eL, status, W, walker0, gen, a, gamma, e_ref,
                                                   max_hops, lw.left, lw.lw, lw.hops, lw.flags, lw.active, lw.moved,
                                                   lw.list_up, lw.list_dn, lw.list_w, lw.cnt);
  return cudaGetLastError();
}

cudaError_t launch_lrdmc_rows(const DevSystem &s, const double *r, const int *moved, double *pprop, double *phi_up,
                              int W, cudaStream_t st) {
  if (W <= 0) return cudaSuccess;
  k_lrdmc_rows<<<W, 128, 0, st>>>(s, r, moved, pprop, phi_up);
  return cudaGetLastError();
}

cudaError_t launch_walker_copy(const WalkerCopies &cp, const int *list, int Wc, bool scatter, cudaStream_t st) {
  if (Wc <= 0 || cp.n <= 0) return cudaSuccess;
  for (int a = 0; a < cp.n; ++a)
    if (cp.c[a].bytes % 4) return cudaErrorInvalidValue;
  k_walker_copy<<<dim3(Wc, cp.n), 256, 0, st>>>(cp, list, scatter ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_lrdmc_finish(int W, const double *lw, const double *eL_cur, double *weight, double *eL_out,
                                cudaStream_t st) {
  if (W <= 0) return cudaSuccess;
  k_lrdmc_finish<<<(W + 127) / 128, 128, 0, st>>>(W, lw, eL_cur, weight, eL_out);
  return cudaGetLastError();
}

cudaError_t launch_lrdmc_branch(int W, int N, uint32_t gen, uint32_t key0, uint32_t key1, double *weight,
                                const double *eL, double *run, int *parent, double *stats, const double *r_old,
                                double *r_new, cudaStream_t st) {
  if (W <= 0) return cudaSuccess;
  k_lrdmc_select<<<1, kSelectThreads, 0, st>>>(W, gen, key0, key1, weight, eL, run, parent, stats);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const long tot = (long)W * N * 3;
  k_lrdmc_gather<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(r_old, parent, W, 3 * N, r_new);
  return cudaGetLastError();
}

cudaError_t launch_lrdmc_energy(const double *wbar, const double *ebar, int T, int p, double *E, cudaStream_t st) {
  k_lrdmc_energy<<<1, 32, 0, st>>>(wbar, ebar, T, p, E);
  return cudaGetLastError();
}

}  // namespace jagp
