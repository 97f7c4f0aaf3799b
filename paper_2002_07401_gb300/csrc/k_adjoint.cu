// k_adjoint.cu -- reverse-mode derivatives (Sec. "Derivatives of energy":
// algorithmic adjoint differentiation) of log|Psi| and of the local energy
// with respect to the pairing matrix lambda, the Jastrow parameters, the
// nuclear positions R_a and the electron positions r_i, for the force of
// Eq. forces:aad (without the space warp).
//
// Notation per walker: Bt_j = lambda phi(r_j^dn) (then the unpaired orbitals),
// A_i = lambda^T phi(r_i^up), G~ = Phi_up Bt^T, M_e the kinetic contraction
// vector of electron e (M_i = sum_j Ginv[j][i] Bt_j, M_{n+j} = sum_i Ginv[j][i] A_i),
// gD_e = grad phi(r_e)^T M_e, lD_e = lap phi(r_e) . M_e.  With seeds sL (on
// log|Psi|) and sE (on e_L) the adjoints are
//   Mbar_e = sE (-1/2 lap phi(r_e) - grad phi(r_e) . grad J_e)
//   H_ij   = Mbar_i . Bt_j + A_i . Mbar_{n+j}
//   Gbar   = -(Ginv H Ginv)^T + sL Ginv^T
//   Btbar_j = sum_i Gbar_ij phi_i + sum_i Ginv_ji Mbar_i,   Abar_i = sum_j Ginv_ji Mbar_{n+j}
//   phibar_i = sum_j Gbar_ij Bt_j + lambda Abar_i (up),     phibar_{n+j} = lambda^T Btbar_j (down)
//   lambdabar = sum_j Btbar_j phi_{n+j}^T + sum_i phi_i Abar_i^T
// and the orbital tables carry them to the positions through the orbital
// gradients, Hessians and gradients of the Laplacian.
#include <math.h>

#include <algorithm>

#include "jagp_launch.h"

namespace jagp {

// ---------------------------------------------------------------------------
// The angular polynomials P_c of a shell are harmonic and homogeneous of degree
// l, so sums over its components need only their coefficients' polynomial and
// its derivatives.  For S = sum_c m_c P_c: value, gradient, and (with b) the
// product of its constant Hessian with a vector.
// ---------------------------------------------------------------------------
struct ShellPoly {
  double v, g[3];
};
__device__ __forceinline__ ShellPoly shell_poly(int l, const double m[5], double x, double y, double z) {
  ShellPoly s;
  if (l == 0) {
    s.v = m[0];
    s.g[0] = s.g[1] = s.g[2] = 0.0;
  } else if (l == 1) {
    s.g[0] = m[0];
    s.g[1] = m[1];
    s.g[2] = m[2];
    s.v = m[0] * x + m[1] * y + m[2] * z;
  } else {
    // xy, yz, zx, x^2 - y^2, 2 z^2 - x^2 - y^2; S = (x S_x + y S_y + z S_z) / 2
    s.g[0] = m[0] * y + m[2] * z + 2.0 * (m[3] - m[4]) * x;
    s.g[1] = m[0] * x + m[1] * z - 2.0 * (m[3] + m[4]) * y;
    s.g[2] = m[1] * y + m[2] * x + 4.0 * m[4] * z;
    s.v = 0.5 * (s.g[0] * x + s.g[1] * y + s.g[2] * z);
  }
  return s;
}

// Radial factor g (e^{-zeta r^2} or e^{-zeta r}) through what its derivatives need:
// grad g = -al g d, lap(P g) = P g h for degree l, grad h = et d, and be with
// grad al = -be d (0 for a Gaussian).
struct Radial {
  double g, al, h, et, be;
};
__device__ __forceinline__ Radial radial_parts(int rad, int l, double zeta, double r2) {
  Radial p;
  if (rad) {
    const double ri = rsqrt(r2), r = r2 * ri, zr = zeta * ri, zr3 = zr * ri * ri;
    p.g = exp(-zeta * r);
    p.al = zr;
    p.h = zeta * zeta - 2.0 * (l + 1) * zr;
    p.et = 2.0 * (l + 1) * zr3;
    p.be = zr3;
  } else {
    p.g = exp(-zeta * r2);
    p.al = 2.0 * zeta;
    p.h = 4.0 * zeta * zeta * r2 - (4 * l + 6) * zeta;
    p.et = 8.0 * zeta * zeta;
    p.be = 0.0;
  }
  return p;
}

// ---------------------------------------------------------------------------
// Jastrow derivatives of one radial function F(r), r = |d|: the first three.
// J1 term of an atom: F = -c^3 u(c r), u = (1 - e^{-b s}) / (2b);
// J2 pair term: F = r / (k (1 + b r)).
// ---------------------------------------------------------------------------
// (and dF/db of the J1 term)
__device__ __forceinline__ void j1_d3(double c, double b, double r, double *f1, double *f2, double *f3, double *fb) {
  const double c3 = c * c * c, c4 = c3 * c, s = c * r;
  if (b == 0.0) {
    *f1 = -0.5 * c4;
    *f2 = 0.0;
    *f3 = 0.0;
    *fb = 0.25 * c3 * s * s;
    return;
  }
  const double e = exp(-b * s), ib = 0.5 / b;
  *f1 = -0.5 * c4 * e;
  *f2 = -c * b * *f1;
  *f3 = -c * b * *f2;
  *fb = -c3 * ib * (s * e - (1.0 - e) * 2.0 * ib);
}
__device__ __forceinline__ void j2_d3(double ik, double b, double iq, double *v1, double *v2, double *v3) {
  *v1 = ik * iq * iq;  // iq = 1 / (1 + b r), ik = 1 / k
  const double t = b * iq;
  *v2 = -2.0 * t * *v1;
  *v3 = -3.0 * t * *v2;
}

// Hessian-vector product H v and gradient of the Laplacian, gl d with gl =
// (f3 + 2 f2/r - 2 f1/r^2) / r, of F(|d|); ri = 1/r
__device__ __forceinline__ void radial_adj(double f1, double f2, double f3, const double d[3], double ri,
                                           const double v[3], double hv[3], double *gl) {
  const double f1r = f1 * ri, dv = (d[0] * v[0] + d[1] * v[1] + d[2] * v[2]) * ri * ri, q = (f2 - f1r) * dv;
  for (int k = 0; k < 3; ++k) hv[k] = q * d[k] + f1r * v[k];
  *gl = (f3 + 2.0 * (f2 - f1r) * ri) * ri;
}

// lanes per group of a warp that takes n items at a time: the power of two >= n, at most 32
__host__ __device__ inline int group_lanes(int n) {
  int g = 1;
  while (g < n && g < 32) g *= 2;
  return g;
}
__device__ __forceinline__ double group_sum(double v, int g) {
  for (int o = g / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// 1. Jastrow gradient at every electron and the kinetic adjoint vectors
//    Mbar_e = sE (-1/2 lap phi - grad phi . grad J_e); also the orbital values
//    at the down electrons (rows of dnphi).  One warp per electron.  Bound by the
//    FP64 pipe: per component P (-h/2 + al b.d) - grad P . b, b = grad J, times g
//    (1000 walkers of 16 He: 0.53 ms; 0.85 with each component's full gradient and Laplacian).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_adj_kvec(DevSystem s, const double *__restrict__ r,
                                                  const double *__restrict__ sE, double *__restrict__ jg,
                                                  double *__restrict__ kbar, double *__restrict__ dnphi, int W) {
  extern __shared__ double4 sh_geo[];
  int *sh_info = reinterpret_cast<int *>(sh_geo + s.n_shells);
  for (int k = threadIdx.x; k < s.n_shells; k += blockDim.x) {
    sh_geo[k] = s.shell_geo[k];
    sh_info[k] = s.shell_info[k];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const long nwarps = (long)gridDim.x * (blockDim.x >> 5);
  const long total = (long)W * s.N;
  for (long pt = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); pt < total; pt += nwarps) {
    const int w = (int)(pt / s.N), e = (int)(pt % s.N);
    const double *xw = r + (size_t)w * s.N * 3;
    const double ex = xw[3 * e], ey = xw[3 * e + 1], ez = xw[3 * e + 2];
    // grad J_e (lanes over atoms and other electrons)
    double gx = 0.0, gy = 0.0, gz = 0.0;
    if (s.use_j1)
      for (int a = lane; a < s.n_atoms; a += 32) {
        const double dx = ex - s.R[3 * a], dy = ey - s.R[3 * a + 1], dz = ez - s.R[3 * a + 2];
        const double r2 = dx * dx + dy * dy + dz * dz, ri = rsqrt(r2), c = s.c1[a], c4 = c * c * c * c;
        const double fp = -0.5 * c4 * (s.b_ea == 0.0 ? 1.0 : exp(-s.b_ea * c * r2 * ri)) * ri;
        gx += fp * dx;
        gy += fp * dy;
        gz += fp * dz;
      }
    if (s.use_j2)
      for (int k = lane; k < s.N; k += 32) {
        if (k == e) continue;
        const double dx = ex - xw[3 * k], dy = ey - xw[3 * k + 1], dz = ez - xw[3 * k + 2];
        const double r2 = dx * dx + dy * dy + dz * dz, ri = rsqrt(r2);
        double kk, bb;
        j2_params(s, (e < s.n_up) == (k < s.n_up), &kk, &bb);
        const double iq = 1.0 / (1.0 + bb * r2 * ri), vp = (kk == 4.0 ? 0.25 : 0.5) * iq * iq * ri;
        gx += vp * dx;
        gy += vp * dy;
        gz += vp * dz;
      }
    gx = warp_sum(gx);
    gy = warp_sum(gy);
    gz = warp_sum(gz);
    if (lane == 0) {
      jg[pt * 3] = gx;
      jg[pt * 3 + 1] = gy;
      jg[pt * 3 + 2] = gz;
    }
    const double se = sE ? sE[w] : 0.0;
    double *kb = kbar + pt * s.L;
    double *dp = (e >= s.n_up) ? dnphi + ((size_t)w * s.n_up + (e - s.n_up)) * s.L : nullptr;
    for (int k = lane; k < s.n_shells; k += 32) {
      const double4 G = sh_geo[k];
      const int info = sh_info[k], l = shell_l(info), off = shell_off(info);
      const double x = ex - G.x, y = ey - G.y, z = ez - G.z, r2 = x * x + y * y + z * z;
      const Radial p = radial_parts(shell_rad(info), l, G.w, r2);
      const double t = p.al * (gx * x + gy * y + gz * z) - 0.5 * p.h, sg = se * p.g;
      if (l == 0) {
        kb[off] = sg * t;
        if (dp) dp[off] = p.g;
      } else if (l == 1) {
        kb[off] = sg * (x * t - gx);
        kb[off + 1] = sg * (y * t - gy);
        kb[off + 2] = sg * (z * t - gz);
        if (dp) {
          dp[off] = x * p.g;
          dp[off + 1] = y * p.g;
          dp[off + 2] = z * p.g;
        }
      } else {
        const double P[5] = {x * y, y * z, z * x, x * x - y * y, 3.0 * z * z - r2};
        const double xg = x * gx, yg = y * gy;
        const double D[5] = {y * gx + x * gy, z * gy + y * gz, x * gz + z * gx, 2.0 * (xg - yg),
                             4.0 * z * gz - 2.0 * (xg + yg)};
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          kb[off + c] = sg * (P[c] * t - D[c]);
          if (dp) dp[off + c] = P[c] * p.g;
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// 2. Gbar = -(Ginv H Ginv)^T + sL Ginv^T with H = H1 + H2 (H2 only in the
//    first n_dn columns).  One CTA per walker, everything in shared memory.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_adj_gbar(const double *__restrict__ ginv, const double *__restrict__ h1,
                                                  const double *__restrict__ h2, const double *__restrict__ sL, int n,
                                                  int nd, double *__restrict__ gbar) {
  extern __shared__ double sm[];
  const int w = blockIdx.x, tid = threadIdx.x, bs = blockDim.x, nn = n * n;
  double *Gi = sm, *Hm = Gi + nn, *T = Hm + nn;
  const double *gw = ginv + (size_t)w * nn;
  for (int t = tid; t < nn; t += bs) {
    Gi[t] = gw[t];
    const int i = t / n, j = t - i * n;
    Hm[t] = h1[(size_t)w * nn + t] + (j < nd ? h2[(size_t)w * nn + (size_t)i * n + j] : 0.0);
  }
  __syncthreads();
  for (int t = tid; t < nn; t += bs) {  // T = Ginv H
    const int i = t / n, j = t - i * n;
    double a = 0.0;
    for (int k = 0; k < n; ++k) a = fma(Gi[i * n + k], Hm[k * n + j], a);
    T[t] = a;
  }
  __syncthreads();
  const double s = sL ? sL[w] : 0.0;
  for (int t = tid; t < nn; t += bs) {  // Gbar_ij = -(T Ginv)_ji + s Ginv_ji
    const int i = t / n, j = t - i * n;
    double a = 0.0;
    for (int k = 0; k < n; ++k) a = fma(T[j * n + k], Gi[k * n + i], a);
    gbar[(size_t)w * nn + t] = -a + s * Gi[j * n + i];
  }
}

// ---------------------------------------------------------------------------
// 3. row adjoints, per (walker, 64 columns):
//    Btbar_j = sum_i Gbar_ij phi_i + sum_i Ginv_ji Mbar_i        (j < n_dn)
//    Abar_i  = sum_j Ginv_ji Mbar_{n+j}                          (i < n)
//    phibar_i (partial) = sum_j Gbar_ij Bt_j                     (i < n)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_adj_rows(DevSystem s, const double *__restrict__ ginv,
                                                  const double *__restrict__ gbar, const double *__restrict__ phi_up,
                                                  const double *__restrict__ bt, const double *__restrict__ kbar,
                                                  double *__restrict__ btbar, double *__restrict__ abar,
                                                  double *__restrict__ phibar) {
  extern __shared__ double sm[];
  const int n = s.n_up, nd = s.n_dn, N = s.N, L = s.L, nn = n * n;
  const int w = blockIdx.y, c0 = blockIdx.x * 64, tid = threadIdx.x;
  double *Gi = sm, *Gb = Gi + nn, *Ph = Gb + nn, *Bs = Ph + n * 64, *Ku = Bs + n * 64, *Kd = Ku + n * 64;
  for (int t = tid; t < nn; t += 256) {
    Gi[t] = ginv[(size_t)w * nn + t];
    Gb[t] = gbar[(size_t)w * nn + t];
  }
  for (int t = tid; t < n * 64; t += 256) {
    const int j = t >> 6, c = t & 63;
    const bool in = c0 + c < L;
    Ph[t] = in ? phi_up[((size_t)w * n + j) * L + c0 + c] : 0.0;
    Bs[t] = in ? bt[((size_t)w * n + j) * L + c0 + c] : 0.0;
    Ku[t] = in ? kbar[((size_t)w * N + j) * L + c0 + c] : 0.0;
    Kd[t] = (in && j < nd) ? kbar[((size_t)w * N + n + j) * L + c0 + c] : 0.0;
  }
  __syncthreads();
  for (int idx = tid; idx < n * 64; idx += 256) {
    const int i = idx >> 6, c = idx & 63;
    if (c0 + c >= L) continue;
    double pb = 0.0, ab = 0.0, bb = 0.0;
    for (int j = 0; j < n; ++j) pb = fma(Gb[i * n + j], Bs[j * 64 + c], pb);
    for (int j = 0; j < nd; ++j) ab = fma(Gi[j * n + i], Kd[j * 64 + c], ab);
    if (i < nd) {
      for (int k = 0; k < n; ++k) bb = fma(Gb[k * n + i], Ph[k * 64 + c], bb);
      for (int k = 0; k < n; ++k) bb = fma(Gi[i * n + k], Ku[k * 64 + c], bb);
      btbar[((size_t)w * n + i) * L + c0 + c] = bb;
    }
    abar[((size_t)w * n + i) * L + c0 + c] = ab;
    phibar[((size_t)w * n + i) * L + c0 + c] = pb;
  }
}

// ---------------------------------------------------------------------------
// 4. orbital tables -> positions.  Per shell at displacement d, with b =
//    -sE grad J_e, lb = -sE / 2, Q = sum_c phibar_c P_c and S = sum_c M_c P_c,
//      grad(Q g) + Hess(S g) b + lb grad(lap(S g))
//        = g [grad Q + (Hess S) b + (lb h - al b.d) grad S - al S b + ka d],
//      ka = -al (Q + u) + be S b.d + lb S (et - al h),  u = b.grad S - al S b.d
//    goes to the electron and, negated, to the shell's atom.  A lane takes an
//    atom and all its shells (lanes in groups of the next power of two, so that
//    a few atoms leave room for several electrons per warp), so the atoms' sums
//    stay in registers: per-component third derivatives with FP64 atomics in
//    shared memory took 2.2 ms for 1000 walkers of 16 He, these 0.58.  A CTA takes kAdjElectrons
//    electrons of one walker; its per-atom sums go to part[w][blockIdx.x][atom].
// ---------------------------------------------------------------------------
constexpr int kAdjWarps = 8;
constexpr int kAdjElectrons = 32;

__global__ void __launch_bounds__(kAdjWarps * 32) k_adj_positions(
    DevSystem s, const double *__restrict__ r, const double *__restrict__ sE, const double *__restrict__ jg,
    const double *__restrict__ mbuf, const double *__restrict__ phibar_a, const double *__restrict__ phibar_b,
    const double *__restrict__ phibar_dn, double *__restrict__ rbar, double *__restrict__ part) {
  __shared__ double s_re[kAdjElectrons][3];  // electrons' sums over the atoms so far
  __shared__ double s_at[kAdjWarps][32][3];   // a chunk of atoms: each warp's lanes
  const int w = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int e0 = blockIdx.x * kAdjElectrons, ne = min(kAdjElectrons, s.N - e0);
  const int G = group_lanes(s.n_atoms), per = 32 / G;  // electrons of a warp at a time
  const int sub = lane / G, ga = lane - sub * G;
  const double se = sE ? sE[w] : 0.0, lb = -0.5 * se;
  for (int t = tid; t < 3 * kAdjElectrons; t += kAdjWarps * 32) s_re[t / 3][t % 3] = 0.0;
  __syncthreads();
  for (int a0 = 0; a0 < s.n_atoms; a0 += G) {
    const int a = a0 + ga;
    const int k0 = a < s.n_atoms ? s.atom_first[a] : 0, k1 = a < s.n_atoms ? s.atom_first[a + 1] : 0;
    double ra[3] = {0.0, 0.0, 0.0};
    const double Rx = a < s.n_atoms ? s.R[3 * a] : 0.0, Ry = a < s.n_atoms ? s.R[3 * a + 1] : 0.0,
                 Rz = a < s.n_atoms ? s.R[3 * a + 2] : 0.0;
    for (int q0 = warp * per; q0 < ne; q0 += kAdjWarps * per) {
      const int q = q0 + sub, e = e0 + q;
      double c[3] = {0.0, 0.0, 0.0};
      if (q < ne) {
        const size_t pt = (size_t)w * s.N + e;
        const double x = r[pt * 3] - Rx, y = r[pt * 3 + 1] - Ry, z = r[pt * 3 + 2] - Rz;
        const double b[3] = {-se * jg[pt * 3], -se * jg[pt * 3 + 1], -se * jg[pt * 3 + 2]};
        const double r2 = x * x + y * y + z * z, bd = b[0] * x + b[1] * y + b[2] * z;
        const double *M = mbuf + pt * s.L;
        const bool up = e < s.n_up;
        const size_t row = (size_t)w * s.n_up + (up ? e : e - s.n_up);
        const double *pa = (up ? phibar_a : phibar_dn) + row * s.L, *pb = up ? phibar_b + row * s.L : nullptr;
        for (int k = k0; k < k1; ++k) {
          const int sh = s.atom_shells[k], info = s.shell_info[sh], l = shell_l(info), off = shell_off(info);
          double m[5], f[5];
#pragma unroll
          for (int i = 0; i < 5; ++i)
            if (i < 2 * l + 1) {
              m[i] = M[off + i];
              f[i] = pa[off + i] + (pb ? pb[off + i] : 0.0);
            }
          const Radial p = radial_parts(shell_rad(info), l, s.shell_geo[sh].w, r2);
          const ShellPoly S = shell_poly(l, m, x, y, z), Q = shell_poly(l, f, x, y, z);
          double H[3] = {0.0, 0.0, 0.0};  // (Hess S) b
          if (l == 2) {
            H[0] = 2.0 * (m[3] - m[4]) * b[0] + m[0] * b[1] + m[2] * b[2];
            H[1] = m[0] * b[0] - 2.0 * (m[3] + m[4]) * b[1] + m[1] * b[2];
            H[2] = m[2] * b[0] + m[1] * b[1] + 4.0 * m[4] * b[2];
          }
          const double aS = p.al * S.v, u = b[0] * S.g[0] + b[1] * S.g[1] + b[2] * S.g[2] - aS * bd;
          const double cs = lb * p.h - p.al * bd;
          const double ka = S.v * (p.be * bd + lb * (p.et - p.al * p.h)) - p.al * (Q.v + u);
          c[0] += p.g * (Q.g[0] + H[0] + cs * S.g[0] - aS * b[0] + ka * x);
          c[1] += p.g * (Q.g[1] + H[1] + cs * S.g[1] - aS * b[1] + ka * y);
          c[2] += p.g * (Q.g[2] + H[2] + cs * S.g[2] - aS * b[2] + ka * z);
        }
      }
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        ra[t] -= c[t];
        const double v = group_sum(c[t], G);
        if (ga == 0 && q < ne) s_re[q][t] += v;  // (this warp's electrons in every chunk)
      }
    }
    // the chunk's atoms over the CTA's electrons
#pragma unroll
    for (int t = 0; t < 3; ++t) s_at[warp][lane][t] = ra[t];
    __syncthreads();
    for (int t = tid; t < 3 * G; t += kAdjWarps * 32) {
      const int i = t / 3, q = t - 3 * i;
      if (a0 + i < s.n_atoms) {
        double v = 0.0;
        for (int ww = 0; ww < kAdjWarps; ++ww)
          for (int h = 0; h < per; ++h) v += s_at[ww][h * G + i][q];
        part[((size_t)w * gridDim.x + blockIdx.x) * 3 * s.n_atoms + 3 * (a0 + i) + q] = v;
      }
    }
    __syncthreads();
  }
  for (int t = tid; t < 3 * ne; t += kAdjWarps * 32) rbar[((size_t)w * s.N + e0) * 3 + t] = s_re[t / 3][t % 3];
}

// ---------------------------------------------------------------------------
// 5. Jastrow and Coulomb adjoints, Jastrow parameter derivatives.  One CTA per
//    walker.  Electron-atom pairs: lanes on atoms (in groups, as above), a pair's
//    terms added to its electron (over the group) and, negated, to its atom (in
//    the lane); electron-electron pairs: a warp per electron, lanes on the others.
//    rbar[e] += ..., rbar_at[w][a] = ..., jpar[w][3] = ...  Bound by the FP64 pipe:
//    one reciprocal square root and one division per pair (1000 walkers of 16 He:
//    0.31 ms; 1.05 with a thread per electron and atomics for the atoms).
// ---------------------------------------------------------------------------
constexpr int kJasWarps = 8;

__global__ void __launch_bounds__(kJasWarps * 32) k_adj_jastrow(DevSystem s, const double *__restrict__ r,
                                                                const double *__restrict__ sL,
                                                                const double *__restrict__ sE,
                                                                const double *__restrict__ jg,
                                                                const double *__restrict__ kin,
                                                                double *__restrict__ rbar,
                                                                double *__restrict__ rbar_at,
                                                                double *__restrict__ jpar) {
  extern __shared__ double sm[];
  __shared__ double s_at[kJasWarps][32][3];
  __shared__ double red[3][kJasWarps];
  const int w = blockIdx.x, N = s.N, tid = threadIdx.x, bs = kJasWarps * 32, lane = tid & 31, warp = tid >> 5;
  double *xs = sm, *gJb = xs + 3 * N, *re_s = gJb + 3 * N;  // positions; adjoint of grad J_e; electrons' sums
  const double sl = sL ? sL[w] : 0.0, se = sE ? sE[w] : 0.0;
  const double lJb = -0.5 * se;        // adjoint of lap J_e (the same for all e)
  for (int t = tid; t < 3 * N; t += bs) {
    xs[t] = r[(size_t)w * N * 3 + t];
    // gbarJ_e = -sE (gD_e + gJ_e); sL grad J_e from J itself
    const int e = t / 3, q = t - 3 * e;
    const double gj = jg[((size_t)w * N + e) * 3 + q];
    gJb[t] = -se * (kin[((size_t)w * N + e) * 4 + q] + gj);
    re_s[t] = sl * gj;
  }
  __syncthreads();
  double pb_ea = 0.0, pb_para = 0.0, pb_anti = 0.0;
  const int G = group_lanes(s.n_atoms), per = 32 / G, sub = lane / G, ga = lane - sub * G;
  for (int a0 = 0; a0 < s.n_atoms; a0 += G) {
    const int a = a0 + ga;
    const bool have = a < s.n_atoms;
    double ra[3] = {0.0, 0.0, 0.0};
    const double R[3] = {have ? s.R[3 * a] : 0.0, have ? s.R[3 * a + 1] : 0.0, have ? s.R[3 * a + 2] : 0.0};
    const double Z = have ? s.Z[a] : 0.0, c1 = have ? s.c1[a] : 0.0;
    for (int q0 = warp * per; q0 < N; q0 += kJasWarps * per) {
      const int e = q0 + sub;
      double re[3] = {0.0, 0.0, 0.0};
      if (have && e < N) {
        const double d[3] = {xs[3 * e] - R[0], xs[3 * e + 1] - R[1], xs[3 * e + 2] - R[2]};
        const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2], ri = rsqrt(r2);
        const double z3 = se * Z * ri * ri * ri;  // V_ei
        double f1r = 0.0;
#pragma unroll
        for (int q = 0; q < 3; ++q) re[q] = z3 * d[q];
        if (s.use_j1) {
          double f1, f2, f3, fb, hv[3], gl;
          j1_d3(c1, s.b_ea, r2 == 0.0 ? 0.0 : r2 * ri, &f1, &f2, &f3, &fb);  // (dJ/db is finite at the nucleus)
          radial_adj(f1, f2, f3, d, ri, gJb + 3 * e, hv, &gl);
          gl *= lJb;
#pragma unroll
          for (int q = 0; q < 3; ++q) re[q] += hv[q] + gl * d[q];
          pb_ea += sl * fb;
          f1r = sl * f1 * ri;
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) ra[q] -= re[q] + f1r * d[q];
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const double v = group_sum(re[q], G);
        if (ga == 0 && e < N) re_s[3 * e + q] += v;  // (an electron belongs to one warp in every chunk)
      }
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) s_at[warp][lane][q] = ra[q];
    __syncthreads();
    for (int t = tid; t < 3 * G; t += bs) {
      const int i = t / 3, q = t - 3 * i, at = a0 + i;
      if (at < s.n_atoms) {
        double v = 0.0;
        for (int ww = 0; ww < kJasWarps; ++ww)
          for (int h = 0; h < per; ++h) v += s_at[ww][h * G + i][q];
        for (int bb = 0; bb < s.n_atoms; ++bb) {  // V_ii
          if (bb == at) continue;
          const double d[3] = {s.R[3 * at] - s.R[3 * bb], s.R[3 * at + 1] - s.R[3 * bb + 1],
                               s.R[3 * at + 2] - s.R[3 * bb + 2]};
          const double ri = rsqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
          v -= se * s.Z[at] * s.Z[bb] * d[q] * ri * ri * ri;
        }
        rbar_at[((size_t)w * s.n_atoms + at) * 3 + q] = v;
      }
    }
    __syncthreads();
  }
  for (int e = warp; e < N; e += kJasWarps) {
    const double ex = xs[3 * e], ey = xs[3 * e + 1], ez = xs[3 * e + 2];
    const bool eup = e < s.n_up;
    double re[3] = {0.0, 0.0, 0.0};
    for (int k = lane; k < N; k += 32) {
      if (k == e) continue;
      const double d[3] = {ex - xs[3 * k], ey - xs[3 * k + 1], ez - xs[3 * k + 2]};
      const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2], ri = rsqrt(r2);
      double t = -se * ri * ri * ri;  // V_ee
      if (s.use_j2) {
        const bool same = eup == (k < s.n_up);
        double kk, bb, v1, v2, v3, hv[3], gl;
        j2_params(s, same, &kk, &bb);
        const double ik = kk == 4.0 ? 0.25 : 0.5, rr = r2 == 0.0 ? 0.0 : r2 * ri, iq = 1.0 / (1.0 + bb * rr);
        j2_d3(ik, bb, iq, &v1, &v2, &v3);
        const double dg[3] = {gJb[3 * e] - gJb[3 * k], gJb[3 * e + 1] - gJb[3 * k + 1], gJb[3 * e + 2] - gJb[3 * k + 2]};
        radial_adj(v1, v2, v3, d, ri, dg, hv, &gl);
        t += 2.0 * lJb * gl;
#pragma unroll
        for (int q = 0; q < 3; ++q) re[q] += hv[q];
        if (k > e) {
          const double vdb = -r2 * ik * iq * iq;
          if (same && !s.j2_si) pb_para += sl * vdb;
          else pb_anti += sl * vdb;
        }
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) re[q] += t * d[q];
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) re[q] = warp_sum(re[q]);
    if (lane < 3) {
      const double v = lane == 0 ? re[0] : (lane == 1 ? re[1] : re[2]);
      rbar[((size_t)w * N + e) * 3 + lane] += re_s[3 * e + lane] + v;
    }
  }
  // Jastrow parameter adjoints (from log|Psi| only): block sums
  pb_ea = warp_sum(pb_ea);
  pb_para = warp_sum(pb_para);
  pb_anti = warp_sum(pb_anti);
  if (lane == 0) {
    red[0][warp] = pb_ea;
    red[1][warp] = pb_para;
    red[2][warp] = pb_anti;
  }
  __syncthreads();
  if (tid < 3) {
    double a0 = 0.0;
    for (int q = 0; q < kJasWarps; ++q) a0 += red[tid][q];
    jpar[(size_t)w * 3 + tid] = a0;
  }
}

// ---------------------------------------------------------------------------
// 6. per-walker nuclear adjoints: rbar_at[w] += sum of the orbital partials;
//    then the totals over walkers (fixed order) for R and the Jastrow params.
// ---------------------------------------------------------------------------
__global__ void k_adj_reduce_walker(const double *__restrict__ part, int nparts, int n_atoms,
                                    double *__restrict__ rbar_at, int W) {
  const long total = (long)W * n_atoms * 3;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
    const long w = t / (n_atoms * 3), q = t % (n_atoms * 3);
    double a = rbar_at[t];
    for (int p = 0; p < nparts; ++p) a += part[((size_t)w * nparts + p) * 3 * n_atoms + q];
    rbar_at[t] = a;
  }
}

// ---------------------------------------------------------------------------
// 7. lambdabar = sum_rows U[row]^T V[row] for two stacked row sets; split over
//    row ranges (blockIdx.z), partial sums to part[z][L][L].
//    Set 1: U = Btbar rows (w, j < n_dn), V = phi(r_j^dn) rows;
//    set 2: U = Phi_up rows (w, i < n_up), V = Abar rows.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_adj_lambda(const double *__restrict__ btbar,
                                                    const double *__restrict__ dnphi,
                                                    const double *__restrict__ phi_up, const double *__restrict__ abar,
                                                    int W, int n, int nd, int L, int rows_per_z,
                                                    double *__restrict__ part) {
  __shared__ double Us[16][64], Vs[16][64];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
  const long rows1 = (long)W * nd, rows_all = rows1 + (long)W * n;
  const long r0 = (long)blockIdx.z * rows_per_z;
  const long r1 = min(rows_all, r0 + rows_per_z);
  double acc[4][4] = {};
  for (long rb = r0; rb < r1; rb += 16) {
    for (int t = tid; t < 16 * 64; t += 256) {
      const int rr = t >> 6, c = t & 63;
      const long row = rb + rr;
      double u = 0.0, v = 0.0;
      if (row < r1) {
        const double *U, *V;
        if (row < rows1) {
          const long w = row / nd, j = row % nd;
          U = btbar + ((size_t)w * n + j) * L;
          V = dnphi + ((size_t)w * n + j) * L;
        } else {
          const long q = row - rows1, w = q / n, i = q % n;
          U = phi_up + ((size_t)w * n + i) * L;
          V = abar + ((size_t)w * n + i) * L;
        }
        if (m0 + c < L) u = U[m0 + c];
        if (n0 + c < L) v = V[n0 + c];
      }
      Us[rr][c] = u;
      Vs[rr][c] = v;
    }
    __syncthreads();
    for (int k = 0; k < 16; ++k) {
      double a[4], b[4];
      for (int i = 0; i < 4; ++i) a[i] = Us[k][ty + 16 * i];
      for (int j = 0; j < 4; ++j) b[j] = Vs[k][tx + 16 * j];
      for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  double *po = part + (size_t)blockIdx.z * L * L;
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) {
      const int mu = m0 + ty + 16 * i, nu = n0 + tx + 16 * j;
      if (mu < L && nu < L) po[(size_t)mu * L + nu] = acc[i][j];
    }
}

__global__ void k_adj_lambda_sum(const double *__restrict__ part, int nz, int LL, double *__restrict__ out) {
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < LL; t += (long)gridDim.x * blockDim.x) {
    double a = 0.0;
    for (int z = 0; z < nz; ++z) a += part[(size_t)z * LL + t];
    out[t] = a;
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
cudaError_t launch_adj_kvec(const DevSystem &s, const double *r, const double *sE, double *jg, double *kbar,
                            double *dnphi, int W, cudaStream_t st) {
  const long total = (long)W * s.N;
  long blocks = (total + 7) / 8;
  if (blocks > 152 * 16) blocks = 152 * 16;
  const size_t smem = (size_t)s.n_shells * (sizeof(double4) + sizeof(int));
  k_adj_kvec<<<(int)blocks, 256, smem, st>>>(s, r, sE, jg, kbar, dnphi, W);
  return cudaGetLastError();
}

cudaError_t launch_adj_gbar(const double *ginv, const double *h1, const double *h2, const double *sL, int n, int nd,
                            double *gbar, int W, cudaStream_t st) {
  const size_t smem = (size_t)3 * n * n * sizeof(double);
  k_adj_gbar<<<W, 256, smem, st>>>(ginv, h1, h2, sL, n, nd, gbar);
  return cudaGetLastError();
}

cudaError_t launch_adj_rows(const DevSystem &s, const double *ginv, const double *gbar, const double *phi_up,
                            const double *bt, const double *kbar, double *btbar, double *abar, double *phibar, int W,
                            cudaStream_t st) {
  const int n = s.n_up;
  const size_t smem = (size_t)(2 * n * n + 4 * n * 64) * sizeof(double);
  dim3 grid((s.L + 63) / 64, W);
  k_adj_rows<<<grid, 256, smem, st>>>(s, ginv, gbar, phi_up, bt, kbar, btbar, abar, phibar);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// N_up beyond shared-memory staging: the same adjoints of steps 2 and 3 as
// per-walker GEMMs (k_bgemm below) with Gbar kept transposed,
//   GbarT = sL Ginv - (Ginv H) Ginv,
//   Btbar = GbarT Phi_up + Ginv Mbar_up,   Abar = Ginv^T Mbar_dn,
//   phibar = GbarT^T Bt.
// ---------------------------------------------------------------------------
// C[w] = alpha op(A[w]) B[w] (+ C[w] when accumulate), op(A) = A or A^T, all
// row-major: op(A) M x K, B K x N, C M x N.  64 x 64 output tiles, 4 x 4 per
// thread, k in chunks of 16 (the k order of every output is 0, 1, ..., K-1).
template <bool TA>
__global__ void __launch_bounds__(256) k_bgemm(const double *__restrict__ A, size_t sa, int lda,
                                               const double *__restrict__ B, size_t sb, int ldb,
                                               double *__restrict__ C, size_t sc, int ldc, int M, int N, int K,
                                               double alpha, int accumulate) {
  __shared__ double As[16][65];  // As[k][i] = op(A)[i0 + i][k0 + k]
  __shared__ double Bs[16][65];  // Bs[k][c] = B[k0 + k][c0 + c]
  const int w = blockIdx.z, i0 = blockIdx.y * 64, c0 = blockIdx.x * 64, tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const double *Aw = A + (size_t)w * sa, *Bw = B + (size_t)w * sb;
  double acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
  for (int k0 = 0; k0 < K; k0 += 16) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int idx = tid + q * 256;
      double av = 0.0, bv = 0.0;
      if (TA) {  // op(A)[i][k] = A[k][i]: consecutive threads take consecutive i
        const int kk = idx >> 6, i = idx & 63;
        if (k0 + kk < K && i0 + i < M) av = Aw[(size_t)(k0 + kk) * lda + i0 + i];
        As[kk][i] = av;
      } else {   // op(A)[i][k] = A[i][k]: consecutive threads take consecutive k
        const int i = idx >> 4, kk = idx & 15;
        if (k0 + kk < K && i0 + i < M) av = Aw[(size_t)(i0 + i) * lda + k0 + kk];
        As[kk][i] = av;
      }
      const int kk = idx >> 6, c = idx & 63;
      if (k0 + kk < K && c0 + c < N) bv = Bw[(size_t)(k0 + kk) * ldb + c0 + c];
      Bs[kk][c] = bv;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      double xa[4], yb[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) xa[a] = As[kk][ty * 4 + a];
#pragma unroll
      for (int b = 0; b < 4; ++b) yb[b] = Bs[kk][tx * 4 + b];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = fma(xa[a], yb[b], acc[a][b]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int i = i0 + ty * 4 + a;
    if (i >= M) continue;
    double *Cr = C + (size_t)w * sc + (size_t)i * ldc;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int c = c0 + tx * 4 + b;
      if (c >= N) continue;
      Cr[c] = accumulate ? fma(alpha, acc[a][b], Cr[c]) : alpha * acc[a][b];
    }
  }
}

static cudaError_t bgemm(bool ta, const double *A, size_t sa, int lda, const double *B, size_t sb, int ldb, double *C,
                         size_t sc, int ldc, int M, int N, int K, double alpha, int accumulate, int W,
                         cudaStream_t st) {
  if (W <= 0 || M <= 0 || N <= 0) return cudaSuccess;
  dim3 grid((N + 63) / 64, (M + 63) / 64, W);
  if (ta)
    k_bgemm<true><<<grid, 256, 0, st>>>(A, sa, lda, B, sb, ldb, C, sc, ldc, M, N, K, alpha, accumulate);
  else
    k_bgemm<false><<<grid, 256, 0, st>>>(A, sa, lda, B, sb, ldb, C, sc, ldc, M, N, K, alpha, accumulate);
  return cudaGetLastError();
}

// H = H1 + H2 (H2 only in the first n_dn columns), in place in h1; GbarT = sL Ginv
__global__ void k_adj_gbar_init(const double *__restrict__ ginv, double *__restrict__ h1,
                                const double *__restrict__ h2, const double *__restrict__ sL, int n, int nd, int W,
                                double *__restrict__ gbarT) {
  const long nn = (long)n * n, total = (long)W * nn;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
    const int w = (int)(t / nn), j = (int)(t % n);
    if (j < nd) h1[t] += h2[t];
    gbarT[t] = (sL ? sL[w] : 0.0) * ginv[t];
  }
}

cudaError_t launch_adj_rows_gemm(const DevSystem &s, const double *ginv, double *h1, double *h2, const double *sL,
                                 const double *phi_up, const double *bt, const double *kbar, double *gbarT,
                                 double *btbar, double *abar, double *phibar, int W, cudaStream_t st, bool gbar_only) {
  const int n = s.n_up, nd = s.n_dn, N = s.N, L = s.L;
  const size_t nn = (size_t)n * n, nL = (size_t)n * L, NL = (size_t)N * L;
  long blocks = ((long)W * nn + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_adj_gbar_init<<<(int)blocks, 256, 0, st>>>(ginv, h1, h2, sL, n, nd, W, gbarT);
  cudaError_t e = cudaGetLastError();
  // T = Ginv H (into h2), GbarT -= T Ginv
  if (!e) e = bgemm(false, ginv, nn, n, h1, nn, n, h2, nn, n, n, n, n, 1.0, 0, W, st);
  if (!e) e = bgemm(false, h2, nn, n, ginv, nn, n, gbarT, nn, n, n, n, n, -1.0, 1, W, st);
  if (gbar_only) return e;
  // Btbar (rows j < n_dn) = GbarT Phi_up + Ginv Mbar_up
  if (!e && nd > 0) e = bgemm(false, gbarT, nn, n, phi_up, nL, L, btbar, nL, L, nd, L, n, 1.0, 0, W, st);
  if (!e && nd > 0) e = bgemm(false, ginv, nn, n, kbar, NL, L, btbar, nL, L, nd, L, n, 1.0, 1, W, st);
  // Abar = Ginv^T Mbar_dn (zero without down electrons)
  if (!e && nd > 0) e = bgemm(true, ginv, nn, n, kbar + nL, NL, L, abar, nL, L, n, L, nd, 1.0, 0, W, st);
  if (!e && nd == 0) e = cudaMemsetAsync(abar, 0, (size_t)W * nL * sizeof(double), st);
  // phibar = GbarT^T Bt
  if (!e) e = bgemm(true, gbarT, nn, n, bt, nL, L, phibar, nL, L, n, L, n, 1.0, 0, W, st);
  return e;
}

int adj_position_parts(const DevSystem &s) { return (s.N + kAdjElectrons - 1) / kAdjElectrons; }

cudaError_t launch_adj_positions(const DevSystem &s, const double *r, const double *sE, const double *jg,
                                 const double *mbuf, const double *phibar_a, const double *phibar_b,
                                 const double *phibar_dn, double *rbar, double *part, int W, cudaStream_t st) {
  dim3 grid(adj_position_parts(s), W);
  k_adj_positions<<<grid, kAdjWarps * 32, 0, st>>>(s, r, sE, jg, mbuf, phibar_a, phibar_b, phibar_dn, rbar, part);
  return cudaGetLastError();
}

cudaError_t launch_adj_jastrow(const DevSystem &s, const double *r, const double *sL, const double *sE,
                               const double *jg, const double *kin, double *rbar, double *rbar_at, double *jpar, int W,
                               cudaStream_t st) {
  const size_t smem = (size_t)9 * s.N * sizeof(double);
  k_adj_jastrow<<<W, kJasWarps * 32, smem, st>>>(s, r, sL, sE, jg, kin, rbar, rbar_at, jpar);
  return cudaGetLastError();
}

cudaError_t launch_adj_reduce(const double *part, int nparts, int n_atoms, double *rbar_at, const double *jpar,
                              int W, double *dR, double *djas, cudaStream_t st) {
  const long total = (long)W * n_atoms * 3;
  long blocks = (total + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  k_adj_reduce_walker<<<(int)blocks, 256, 0, st>>>(part, nparts, n_atoms, rbar_at, W);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (dR && (e = launch_walker_sum(rbar_at, W, 3 * n_atoms, dR, st)) != cudaSuccess) return e;
  if (djas) e = launch_walker_sum(jpar, W, 3, djas, st);
  return e;
}

static int adj_lambda_rows_per_z(long rows, int nz) { return (int)(((rows + nz - 1) / nz + 15) / 16 * 16); }

int adj_lambda_most_splits(int W, int n, int nd, int L) {
  const long rows = (long)W * (n + nd), tiles = (long)((L + 63) / 64) * ((L + 63) / 64);
  const long few = std::min(rows / 64, (8 * 152 + tiles - 1) / tiles);
  return (int)std::max(1l, std::min(64l, std::max(rows / 1024, few)));
}

int adj_lambda_splits(int W, int n, int nd, int L) {
  const long rows = (long)W * (n + nd), tiles = (long)((L + 63) / 64) * ((L + 63) / 64);
  const int most = adj_lambda_most_splits(W, n, nd, L);
  int best = most;
  long least = 0;
  for (int nz = most; nz >= 1 && (nz == most || tiles * nz > 3 * 152); --nz) {
    const long c = ((tiles * nz + 151) / 152) * (adj_lambda_rows_per_z(rows, nz) + 8);
    if (nz == most || c <= least) best = nz, least = c;
  }
  return best;
}

cudaError_t launch_adj_lambda(const double *btbar, const double *dnphi, const double *phi_up, const double *abar,
                              int W, int n, int nd, int L, double *part, int nz, double *dlam, cudaStream_t st) {
  const long rows = (long)W * (n + nd);
  const int rows_per_z = adj_lambda_rows_per_z(rows, nz);
  dim3 grid((L + 63) / 64, (L + 63) / 64, nz);
  k_adj_lambda<<<grid, 256, 0, st>>>(btbar, dnphi, phi_up, abar, W, n, nd, L, rows_per_z, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const long LL = (long)L * L;
  long blocks = (LL + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  k_adj_lambda_sum<<<(int)blocks, 256, 0, st>>>(part, nz, (int)LL, dlam);
  return cudaGetLastError();
}

cudaError_t launch_adj_lambda_sum(const double *part, int nz, int L, double *dlam, cudaStream_t st) {
  const long LL = (long)L * L;
  long blocks = (LL + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  k_adj_lambda_sum<<<(int)blocks, 256, 0, st>>>(part, nz, (int)LL, dlam);
  return cudaGetLastError();
}

cudaError_t setup_adjoint_attributes() {
  const int big = 200 * 1024;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_adj_kvec, cudaFuncAttributeMaxDynamicSharedMemorySize, big))) return e;
  if ((e = cudaFuncSetAttribute(k_adj_gbar, cudaFuncAttributeMaxDynamicSharedMemorySize, big))) return e;
  if ((e = cudaFuncSetAttribute(k_adj_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, big))) return e;
  return cudaFuncSetAttribute(k_adj_jastrow, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
}

}  // namespace jagp
