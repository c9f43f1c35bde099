// Reverse-mode derivative (adjoint) of the right-hand side (Sect. 3.1) and of
// the predictor-corrector update (Sect. 3.4.1), in FP64, with the partner
// lists and the damage of the forward evaluation held fixed.
//
// Given cotangents of the right-hand side's outputs (dx/dt, dv/dt, drho/dt,
// du/dt, dS/dt) the kernels accumulate the cotangents of the state (x, v,
// rho, u, S) and of the material parameters (shear modulus mu, yield stress
// Y0, bulk modulus K: a common scale of K0, A_T and B_T).  Every pair term of
// particle a depends on both a and its partner b; because the lists are
// symmetric (b in N(a) iff a in N(b)) each particle gathers, over its own
// list, both the derivatives of its own terms and the derivatives of its
// partners' terms with respect to itself.  No atomics, deterministic order.
//
//   k_adj_passB   reverse of the momentum / energy pass -> x, v, T, c_s, rho
//   k_adj_update  from the forward's pass-A sums, reverse of the constitutive update
//                 (T = sigma/rho^2, damage-reduced stress, Hooke + Jaumann,
//                 von Mises, EOS, grad v = G C with C = L^-1) -> S, u, rho,
//                 parameters, and the cotangents of the pass-A sums
//   k_adj_passA   reverse of the continuity / L / G / XSPH sums -> x, v, rho
//
// Not covered (argument error): artificial stress, density by kernel sum,
// gravity.  Branch switches (viscosity on/off, yield on/off, EOS branches,
// C = I fallback) are held at the forward evaluation's side.
#include "eos.cuh"
#include "fpbits.cuh"
#include "pairs64.cuh"
#include "sph_internal.cuh"

namespace sph {

struct AdjArgs {
  int dim;
  int64_t n, ld;
  const double *x[3], *v[3], *rho, *u, *m, *h, *S, *dmg;
  const int32_t *mat;
  const int32_t *nb_idx, *nb_cnt;
  const double *T, *cs;               // forward pass A (FP64, stride ld)
  const double *bdx[3], *bdv[3], *bdrho, *bdu, *bdS;  // output cotangents
  double *gx[3], *gv[3], *grho, *gu, *gS;             // accumulated state cotangents
  double *Tbar, *csbar;               // scratch: 6 * ld, ld
  double *inter;                      // scratch: 22 * ld (sum_rho_bar, Lbar 9, Gbar 9, xsph_bar 3)
  double *pbar;                       // scratch: 3 * ld (mu, Y0, K per particle)
  MatTable mt;
  sph_params prm;
  // mixed mode: FP32 views and code units of the forward evaluation
  PackedF32 pk;
  const float4 *Tf;                   // forward pass A: (T0..T3), (T4, T5, c_s, 0) in code units
  float4 *Bpk;                        // output cotangents of dv and du in code units (ld)
  float4 *Apk;                        // cotangents of the pass-A sums in code units (6 * ld)
  const Units *U;
  const float *sums;  // mixed: the forward pass A's pair sums (16 rows of stride ld)
  int lane_shift;     // FP64: 2^lane_shift lanes share a particle's partner list
  // mixed: the viscosity parameters in FP32, converted on the host (in the pair
  // loop the compiler converted them for every pair, three FP64-unit
  // instructions)
  float f_alpha, f_beta, f_eps_v;
};

// Conversions of the mixed reverse on the integer pipe (fpbits.cuh), exact or
// rounded as the FP64-unit instructions would; F = double passes values through.
template <class F>
__device__ __forceinline__ F narrow(double v) {
  if constexpr (sizeof(F) == 4) return to_f32_scaled(v, 0, 1.0);
  else return v;
}
// v * sc for a power of two sc
template <class F>
__device__ __forceinline__ F narrow(double v, double sc) {
  if constexpr (sizeof(F) == 4) return to_f32_scaled(v, pow2_exp(sc), sc);
  else return v;
}
__device__ __forceinline__ double widen(float v, double sc) { return to_f64_scaled(v, pow2_exp(sc), sc); }
__device__ __forceinline__ double widen(double v, double) { return v; }
// N values at once with one fallback branch: a call per value (to_f32_scaled's)
// would make the compiler save its live registers around each
template <int N, class F>
__device__ __forceinline__ void narrow_n(const double *v, double sc, F *out) {
  if constexpr (sizeof(F) == 4) {
    const int k = pow2_exp(sc);
    bool ok = true;
#pragma unroll
    for (int i = 0; i < N; ++i) ok &= f32_rn_scaled(v[i], k, out[i]);
    if (!ok) {
#pragma unroll
      for (int i = 0; i < N; ++i) out[i] = __double2float_rn(v[i] * sc);
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) out[i] = v[i];
  }
}
// f *= sc in FP32, sc a power of two: one rounding, of the exact product, as in
// FP64 and back
template <int N>
__device__ __forceinline__ void shift_n(float *f, double sc) {
  const int k = pow2_exp(sc);
  if (k >= -126 && k <= 127) {
    const float fs = bitsf((uint32_t)(k + 127) << 23);
#pragma unroll
    for (int i = 0; i < N; ++i) f[i] *= fs;
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) f[i] = __double2float_rn((double)f[i] * sc);
  }
}

__device__ __forceinline__ int sidx(int dim, int i, int j) { return symk(dim, i, j); }

// Partner list of particle c in the mixed pair kernels: the index read two
// pairs ahead and the partner's position views one pair ahead (as in the
// forward pass A), so that their loads are in flight during the pair before.
struct AdjCursor {
  const int32_t *col;
  int64_t ld;
  int cnt;
  int32_t e1, e2;
  float4 P1, Q1;
  __device__ __forceinline__ void start(const AdjArgs &A, int64_t c, int n) {
    col = A.nb_idx + c;
    ld = A.ld;
    cnt = n;
    e1 = n > 0 ? col[0] : 0;
    e2 = n > 1 ? col[ld] : 0;
    if (n > 0) {
      P1 = A.pk.px(e1);
      Q1 = A.pk.pxl(e1);
    }
  }
  __device__ __forceinline__ int32_t next(const AdjArgs &A, int k, float4 &P, float4 &Q) {
    const int32_t e = e1;
    P = P1;
    Q = Q1;
    e1 = e2;
    if (k + 2 < cnt) e2 = col[(int64_t)(k + 2) * ld];
    if (k + 1 < cnt) {
      P1 = A.pk.px(e1);
      Q1 = A.pk.pxl(e1);
    }
    return e;
  }
};

// Kernel radial factors for a pair: phi = dW/dr / r and phi'(r)/r, W, dW/dr.
template <class R>
struct KPair {
  R phi, dphi_r, W, dWdr;
};

template <class R>
__device__ __forceinline__ KPair<R> kernel_pair(int dim, R r, R hab) {
  const R sig = kernel_sigma<R>(dim);
  const R hinv = R(1.0) / hab;
  const R hD = hpow(hinv, dim);
  const R gnorm = R(6.0) * sig * hD * hinv;
  const R q = r * hinv;
  R s = R(0.0), sp = R(0.0), w = R(0.0);
  if (q < R(0.5)) {
    s = R(3.0) * q * q - R(2.0) * q;
    sp = R(6.0) * q - R(2.0);
    w = R(6.0) * q * q * q - R(6.0) * q * q + R(1.0);
  } else if (q <= R(1.0)) {
    const R t = R(1.0) - q;
    s = -t * t;
    sp = R(2.0) * t;
    w = R(2.0) * t * t * t;
  }
  KPair<R> k;
  k.dWdr = gnorm * s;
  k.W = sig * hD * w;
  const R d2W = gnorm * sp * hinv;
  if (r > R(0.0)) {
    const R ir = R(1.0) / r;
    k.phi = k.dWdr * ir;
    k.dphi_r = (d2W - k.phi) * ir * ir;
  } else {
    k.phi = -R(2.0) * gnorm * hinv;  // limit of dW/dr / r at r = 0
    k.dphi_r = R(0.0);
  }
  return k;
}

// ---------------------------------------------------------------------------
// Reverse of one momentum/energy pair term of particle a with partner b:
//   dv_a += m_b B g,  du_a += -1/2 m_b w.(B g),  B = T_a + T_b - Pi I,  g = phi d
// Given the cotangents vb (of dv_a) and ub (of du_a), returns the cotangents
// of d = x_a - x_b, w = v_a - v_b, of B (symmetrised; it goes to T_a and T_b),
// and half the cotangents of the pair's mean sound speed and density.
// ---------------------------------------------------------------------------
// Artificial viscosity of a pair and its partial derivatives; symmetric in
// the two particles (v.r, the mean sound speed and density do not change when
// they swap), so computed once for both terms of the pair.
template <class R>
struct VPair {
  R vx, Pi, dPi_dnu, dnu_dvx, dnu_dr2, dPi_dc, dPi_drb;
};

template <class R>
__device__ __forceinline__ VPair<R> visc_pair(int dim, const R d[3], const R w[3], R r2, R hab,
                                              R rho_a, R rho_b, R cs_a, R cs_b,
                                              R alpha, R beta, R eps_v) {
  VPair<R> V;
  V.vx = R(0.0);
  for (int i = 0; i < dim; ++i) V.vx += w[i] * d[i];
  V.Pi = V.dPi_dnu = V.dnu_dvx = V.dnu_dr2 = V.dPi_dc = V.dPi_drb = R(0.0);
  if (V.vx < R(0.0)) {
    const R iQ = R(1.0) / (r2 + eps_v * hab * hab);
    const R nu = hab * V.vx * iQ;
    const R cb = R(0.5) * (cs_a + cs_b), irb = R(1.0) / (R(0.5) * (rho_a + rho_b));
    V.Pi = (-alpha * cb * nu + beta * nu * nu) * irb;
    V.dPi_dnu = (-alpha * cb + R(2.0) * beta * nu) * irb;
    V.dnu_dvx = hab * iQ;
    V.dnu_dr2 = -nu * iQ;
    V.dPi_dc = -alpha * nu * irb;
    V.dPi_drb = -V.Pi * irb;
  }
  return V;
}

// K: the kernel factors of the pair (the same for both of its terms); Vs: its
// artificial viscosity (the same for both terms: v.r is unchanged when d and
// w change sign together).
template <class R>
__device__ void pairB_adj(int dim, const R d[3], const R w[3], const KPair<R> &K, const VPair<R> &Vs,
                          const R Ta[6], const R Tb[6], R mb, const R vb[3], R ub,
                          R dbar[3], R wbar[3], R Bsym[6], R &cs_half, R &rho_half) {
  const int ns = nsym(dim);
  R g[3] = {0, 0, 0};
  for (int i = 0; i < dim; ++i) g[i] = K.phi * d[i];
  const R vx = Vs.vx, Pi = Vs.Pi, dPi_dnu = Vs.dPi_dnu, dnu_dvx = Vs.dnu_dvx, dnu_dr2 = Vs.dnu_dr2,
               dPi_dc = Vs.dPi_dc, dPi_drb = Vs.dPi_drb;
  R B[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      if (i < dim && j < dim) {
        const int k = sidx(dim, i, j);
        B[i][j] = Ta[k] + Tb[k] - (i == j ? Pi : R(0.0));
      } else {
        B[i][j] = R(0.0);
      }
    }
  R Bg[3] = {0, 0, 0}, Bw[3] = {0, 0, 0}, Bv[3] = {0, 0, 0};
  for (int i = 0; i < dim; ++i)
    for (int j = 0; j < dim; ++j) {
      Bg[i] += B[i][j] * g[j];
      Bw[i] += B[i][j] * w[j];
      Bv[i] += B[i][j] * vb[j];
    }
  // cotangents of B (general matrix), g and w
  R Bbar[3][3];
  R trB = R(0.0);
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      Bbar[i][j] = (i < dim && j < dim) ? mb * vb[i] * g[j] - R(0.5) * mb * ub * w[i] * g[j] : R(0.0);
      if (i == j) trB += Bbar[i][j];
    }
  R gbar[3] = {0, 0, 0};
  for (int i = 0; i < 3; ++i) {
    gbar[i] = mb * Bv[i] - R(0.5) * mb * ub * Bw[i];
    wbar[i] = -R(0.5) * mb * ub * Bg[i];
    dbar[i] = R(0.0);
  }
  for (int i = 0; i < dim; ++i)
    for (int j = i; j < dim; ++j) Bsym[sidx(dim, i, j)] = R(0.5) * (Bbar[i][j] + Bbar[j][i]);
  for (int k = ns; k < 6; ++k) Bsym[k] = R(0.0);
  cs_half = R(0.0);
  rho_half = R(0.0);
  if (vx < R(0.0)) {
    const R Pibar = -trB;
    const R nubar = Pibar * dPi_dnu;
    const R vxbar = nubar * dnu_dvx;
    const R r2bar = nubar * dnu_dr2;
    cs_half = R(0.5) * Pibar * dPi_dc;
    rho_half = R(0.5) * Pibar * dPi_drb;
    for (int i = 0; i < dim; ++i) {
      wbar[i] += vxbar * d[i];
      dbar[i] += vxbar * w[i] + R(2.0) * r2bar * d[i];
    }
  }
  R gd = R(0.0);
  for (int i = 0; i < dim; ++i) gd += gbar[i] * d[i];
  for (int i = 0; i < dim; ++i) dbar[i] += K.phi * gbar[i] + K.dphi_r * gd * d[i];
}

__device__ __forceinline__ void load_T64(const AdjArgs &A, int64_t a, double t[6]) {
  const int ns = nsym(A.dim);
  for (int k = 0; k < 6; ++k) t[k] = k < ns ? A.T[(int64_t)k * A.ld + a] : 0.0;
}

// FP64, per dimension (every small-matrix loop has a compile-time bound and the
// matrices stay in registers).  Both terms of a pair are one bilinear form in
// d and w: with y = m_e vb_c - m_c vb_e - (m_e ub_c + m_c ub_e) w / 2 the sum of
// the two is phi y.(B d), so that one product B d, one B y and one outer
// product give every cotangent of the pair.  Bound by the FP64 unit; about 150
// FP64 instructions a pair where evaluating the two terms one after the other,
// with their divisions, took 490 (33k particles: 1.40 -> 0.50 ms).
template <int DIM>
__global__ void k_adj_passB(AdjArgs A) {
  const int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> A.lane_shift;
  if (c >= A.n) return;
  const Lanes64 ln(A.lane_shift);
  constexpr int NS = DIM == 3 ? 6 : 3;
  const sph_params &P = A.prm;
  double xc[DIM], vc[DIM], vbc[DIM], Tc[6];
#pragma unroll
  for (int i = 0; i < DIM; ++i) {
    xc[i] = A.x[i][c];
    vc[i] = A.v[i][c];
    vbc[i] = A.bdv[i] ? A.bdv[i][c] : 0.0;
  }
  const double ubc = A.bdu ? A.bdu[c] : 0.0;
  load_T64(A, c, Tc);
  const double rc = A.rho[c], csc = A.cs[c], mc = A.m[c];
  Support64<DIM> H;
  H.start(A.h[c]);
  double gx[DIM], gv[DIM], Tb[6], csbar = 0.0, rhobar = 0.0;
#pragma unroll
  for (int i = 0; i < DIM; ++i) gx[i] = gv[i] = 0.0;
#pragma unroll
  for (int k = 0; k < 6; ++k) Tb[k] = 0.0;
  const int cnt = A.nb_cnt[c];
  for (int k = ln.sub; k < cnt; k += ln.n) {
    const int32_t e = A.nb_idx[(int64_t)k * A.ld + c];
    const double me = A.m[e];
    const double U = 0.5 * fma(me, ubc, A.bdu ? mc * A.bdu[e] : 0.0);
    double d[3] = {0.0, 0.0, 0.0}, w[3] = {0.0, 0.0, 0.0}, y[3] = {0.0, 0.0, 0.0}, B[6];
    double r2 = 0.0, vx = 0.0, yd = 0.0;
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      d[i] = xc[i] - A.x[i][e];
      w[i] = vc[i] - A.v[i][e];
      y[i] = fma(-U, w[i], fma(me, vbc[i], A.bdv[i] ? -mc * A.bdv[i][e] : 0.0));
      r2 = fma(d[i], d[i], r2);
      vx = fma(w[i], d[i], vx);
      yd = fma(y[i], d[i], yd);
    }
#pragma unroll
    for (int q = 0; q < NS; ++q) B[q] = Tc[q] + A.T[(int64_t)q * A.ld + e];
    H.partner(A.h[e]);
    double phi, dphi, qq;
    radial64(H, r2, phi, dphi, qq);
    double vxb = 0.0, r2b = 0.0;  // cotangents of v.r and (twice) r^2 through the viscosity
    if ((int64_t)dbits(vx) < 0) {
      const double iQ = rcp64(fma(P.eps_v * H.hab, H.hab, r2)), irb = rcp64(rc + A.rho[e]);
      const double nu = H.hab * vx * iQ, cb = P.alpha * (csc + A.cs[e]), b2 = 2.0 * P.beta * nu;
      const double Pi = nu * (b2 - cb) * irb;  // = (-alpha c nu + beta nu^2) / rho, c and rho means
#pragma unroll
      for (int i = 0; i < DIM; ++i) B[i] -= Pi;
      const double pib = -phi * yd;  // cotangent of Pi
      const double nub = pib * (2.0 * b2 - cb) * irb;
      vxb = nub * H.hab * iQ;
      r2b = -2.0 * nub * nu * iQ;
      csbar = fma(-pib * P.alpha, nu * irb, csbar);
      rhobar = fma(-pib, Pi * irb, rhobar);
    }
    double s[3], t[3];
    sym_mv(DIM, B, d, s);
    sym_mv(DIM, B, y, t);
    double Fs = 0.0;
#pragma unroll
    for (int i = 0; i < DIM; ++i) Fs = fma(y[i], s[i], Fs);
    const double cd = fma(dphi, Fs, r2b), cw = -U * phi;
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      gx[i] += fma(phi, t[i], fma(cd, d[i], vxb * w[i]));
      gv[i] += fma(cw, s[i], vxb * d[i]);
      y[i] *= phi;
    }
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
      for (int j = i; j < DIM; ++j) {
        const int q = symk(DIM, i, j);
        Tb[q] = fma(y[i], d[j], Tb[q]);
        if (j > i) Tb[q] = fma(y[j], d[i], Tb[q]);
      }
  }
  const double norm = 6.0 * kernel_sigma<double>(DIM);
#pragma unroll
  for (int i = 0; i < DIM; ++i) {
    gx[i] = norm * ln.sum(gx[i]);
    gv[i] = norm * ln.sum(gv[i]);
  }
#pragma unroll
  for (int q = 0; q < NS; ++q) Tb[q] = (q < DIM ? 1.0 : 0.5) * norm * ln.sum(Tb[q]);
  csbar = norm * ln.sum(csbar);
  rhobar = norm * ln.sum(rhobar);
  if (ln.sub) return;
#pragma unroll
  for (int i = 0; i < DIM; ++i) {
    A.gx[i][c] += gx[i];
    A.gv[i][c] += gv[i];
  }
  A.grho[c] += rhobar;
  for (int q = 0; q < 6; ++q) A.Tbar[(int64_t)q * A.ld + c] = q < NS ? Tb[q] : 0.0;
  A.csbar[c] = csbar;
}

// ---------------------------------------------------------------------------
// Constitutive update, recomputed and reversed
// ---------------------------------------------------------------------------
template <class R>
__device__ __forceinline__ bool invert_L(int dim, const R L[3][3], R C[3][3]) {
  R det;
  if (dim == 2) det = L[0][0] * L[1][1] - L[0][1] * L[1][0];
  else
    det = L[0][0] * (L[1][1] * L[2][2] - L[1][2] * L[2][1]) - L[0][1] * (L[1][0] * L[2][2] - L[1][2] * L[2][0]) +
          L[0][2] * (L[1][0] * L[2][1] - L[1][1] * L[2][0]);
  R diag = R(1);
  for (int i = 0; i < dim; ++i) diag *= fabs(L[i][i]);
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) C[i][j] = i == j ? R(1) : R(0);
  if (!(fabs(det) > R(1e-8) * diag) || !(diag > R(0))) return false;
  const R inv = R(1) / det;
  if (dim == 2) {
    C[0][0] = L[1][1] * inv;
    C[0][1] = -L[0][1] * inv;
    C[1][0] = -L[1][0] * inv;
    C[1][1] = L[0][0] * inv;
    return true;
  }
  C[0][0] = (L[1][1] * L[2][2] - L[1][2] * L[2][1]) * inv;
  C[0][1] = (L[0][2] * L[2][1] - L[0][1] * L[2][2]) * inv;
  C[0][2] = (L[0][1] * L[1][2] - L[0][2] * L[1][1]) * inv;
  C[1][0] = (L[1][2] * L[2][0] - L[1][0] * L[2][2]) * inv;
  C[1][1] = (L[0][0] * L[2][2] - L[0][2] * L[2][0]) * inv;
  C[1][2] = (L[0][2] * L[1][0] - L[0][0] * L[1][2]) * inv;
  C[2][0] = (L[1][0] * L[2][1] - L[1][1] * L[2][0]) * inv;
  C[2][1] = (L[0][1] * L[2][0] - L[0][0] * L[2][1]) * inv;
  C[2][2] = (L[0][0] * L[1][1] - L[0][1] * L[1][0]) * inv;
  return true;
}

// p and c_s of a material whose bulk-modulus constants are scaled by s.
__device__ void eos_scaled(const sph_material &M0, double s, double rho, double u, double &p, double &cs, double *pr,
                           double *pu) {
  sph_material M = M0;
  M.K0 *= s;
  M.A_T *= s;
  M.B_T *= s;
  const EosC<double> K = eos_consts<double>(M, nullptr, nullptr);
  eos_eval<double>(M, K, rho, u, p, cs, pr, pu);
}

// MIXED: the pass-A sums are the forward pass A's own (FP32, code units, kept
// by it for this kernel), the equation of state is differentiated in FP32
// dual numbers, and the rest of the reverse runs in FP32 in SI units.  The
// reverse is linear in the cotangents it is given (of T, c_s and dS/dt), so
// each particle's are scaled by a power of two to order one first and its
// results scaled back exactly: FP32's exponent range then limits only the
// state, whose SI values it holds.  FP64: the sums of the FP64 pass A, and the
// reverse is FP64 throughout (F = double, no scaling).  The mixed form was bound
// by the FP64 unit (76 % of it) through its conversions; on the integer pipe, and
// writing pass A's cotangents in code units itself, it and the kernels around it
// take 0.47 instead of 0.53 ms at 1M (five blocks per SM; 3 % of the call slower
// at the compiler's 131 registers).
template <bool MIXED, int DIM>
__global__ void __launch_bounds__(128, MIXED ? 5 : 1) k_adj_update(AdjArgs A) {
  using F = typename std::conditional<MIXED, float, double>::type;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= A.n) return;
  constexpr int dim = DIM;
  const int ns = nsym(dim);
  const sph_params &P = A.prm;
  const int64_t ld = A.ld;
  // ---- pass-A sums ----
  const double rc = A.rho[c];
  double srho = 0.0;
  F L[3][3], G[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) L[i][j] = G[i][j] = F(0);
  const int cnt = A.nb_cnt[c];
  {
    // k_passA's KEEP_SUMS layout; the continuity sum and G are rates (mixed:
    // code unit 1/T, a power of two, so that the conversion is exact), L is a
    // number.  FP64: the rows this kernel overwrites at its end.
    const F *sm;
    if constexpr (MIXED) sm = A.sums;
    else sm = A.inter;
    const F it = MIXED ? narrow<F>(A.U->invT) : F(1);
    srho = MIXED ? widen(sm[c], A.U->invT) : (double)sm[c];
    for (int i = 0; i < dim; ++i)
      for (int j = 0; j <= i; ++j) L[i][j] = L[j][i] = sm[(int64_t)(1 + i * (i + 1) / 2 + j) * ld + c];
    for (int i = 0; i < dim; ++i)
      for (int j = 0; j < dim; ++j) G[i][j] = sm[(int64_t)(7 + 3 * i + j) * ld + c] * it;
  }
  F C[3][3];
  const bool corr = P.consistency && cnt >= dim + 1 && invert_L<F>(dim, L, C);
  if (!corr)
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) C[i][j] = i == j ? F(1) : F(0);
  F gv[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      F s = F(0);
      for (int k = 0; k < dim; ++k) s += G[i][k] * C[k][j];
      gv[i][j] = (i < dim && j < dim) ? s : F(0);
    }
  // ---- constitutive state ----
  const int mi0 = A.mat ? A.mat[c] : 0;
  const int mi = (mi0 >= 0 && mi0 < A.mt.nmat) ? mi0 : 0;
  const sph_material &M = A.mt.m[mi];
  const double uc = A.u[c];
  const F mu = narrow<F>(M.mu), Y0 = narrow<F>(M.Y0);
  F p, pr, pu;
  // MIXED: one evaluation in FP32 dual numbers, in the forward's code units,
  // gives p, dp/drho, dp/du and the exact derivatives of c_s in rho and u and
  // of p and c_s in the bulk-modulus scale (code units to SI by powers of
  // two); FP64: the analytic derivatives of p here, those of c_s and the
  // scale by central differences below.
  F dcr = F(0), dcu = F(0), dps = F(0), dcs = F(0);
  if constexpr (MIXED) {
    const Units *U = A.U;
    const EosC<ad::Dual3> K = eos_consts<ad::Dual3>(M, U->matf[mi], U);
    ad::Dual3 p3, c3, pr3, pu3;
    eos_eval<ad::Dual3>(M, K, rc, uc, p3, c3, &pr3, &pu3);
    const float sig = narrow<float>(U->sig), V = narrow<float>(U->V);
    p = p3.v * sig;
    pr = pr3.v * narrow<float>(U->sig, U->invrho);
    pu = pu3.v * narrow<float>(U->sig, U->invE);
    dcr = c3.d[0] * narrow<float>(U->V, U->invrho);
    dcu = c3.d[1] * narrow<float>(U->V, U->invE);
    dps = p3.d[2] * sig;
    dcs = c3.d[2] * V;
  } else {
    double cs;
    eos_scaled(M, 1.0, rc, uc, p, cs, &pr, &pu);
  }
  const bool strength = A.S != nullptr && M.strength;
  F S[3][3], St[3][3];
  {
    double s64[6];
    F s6[6];
    for (int k = 0; k < 6; ++k) s64[k] = strength && k < ns ? A.S[(int64_t)k * A.n + c] : 0.0;
    narrow_n<6>(s64, 1.0, s6);
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) S[i][j] = (i < dim && j < dim) ? s6[sidx(dim, i, j)] : F(0);
  }
  F J2 = F(0);
  for (int i = 0; i < dim; ++i)
    for (int j = 0; j < dim; ++j) J2 += S[i][j] * S[i][j];
  J2 *= F(0.5);
  F fY = F(1);
  if (strength && M.Y0 > 0.0 && J2 > F(0)) {
    const F q = Y0 * Y0 / (F(3) * J2);
    fY = q < F(1) ? q : F(1);
  }
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) St[i][j] = fY * S[i][j];
  const bool damage = A.dmg != nullptr && M.damage;
  F dd = F(0);
  if (damage) {
    const F del = narrow<F>(A.dmg[c]);
    dd = del * del * del;
  }
  // ---- the cotangents (of T, c_s, dS/dt), scaled (MIXED) ----
  double sc = 1.0, isc = 1.0;
  if constexpr (MIXED) {
    // the largest magnitude, from the bits (a NaN does not count)
    const uint64_t inf = 0x7ff0000000000000ULL;
    uint64_t mx = 0;
    auto largest = [&](double v) {
      const uint64_t b = dbits(v) & 0x7fffffffffffffffULL;
      if (b > mx && b <= inf) mx = b;
    };
    largest(A.csbar[c]);
    for (int k = 0; k < ns; ++k) largest(A.Tbar[(int64_t)k * ld + c]);
    if (A.bdS && strength)
      for (int k = 0; k < ns; ++k) largest(A.bdS[(int64_t)k * A.n + c]);
    const int e = (int)(mx >> 52) - 1022;  // 2^(e-1) <= mx < 2^e for a normal number
    if (e > -1022 && e < 1024) {
      sc = bitsd((uint64_t)(1023 - e) << 52);
      isc = bitsd((uint64_t)(1023 + e) << 52);
    } else if (mx > 0 && mx < inf) {
      int es;
      frexp(bitsd(mx), &es);
      sc = ldexp(1.0, -es);
      isc = ldexp(1.0, es);
    }
  }
  // ---- reverse: T = sigma / rho^2 ----
  F Tb[3][3], Tc[6];
  {
    if constexpr (MIXED) {
      const float4 t0 = A.Tf[c], t1 = A.Tf[ld + c];
      const float t[6] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y};
      for (int k = 0; k < 6; ++k) Tc[k] = k < ns ? t[k] : 0.f;
      shift_n<6>(Tc, A.U->sig * A.U->invrho * A.U->invrho);  // T = sigma / rho^2
    } else {
      load_T64(A, c, Tc);
    }
  }
  F TbT = F(0), trSig = F(0);
  {
    double t64[6];
    F t6[6];
    for (int k = 0; k < 6; ++k) t64[k] = k < ns ? A.Tbar[(int64_t)k * ld + c] : 0.0;
    narrow_n<6>(t64, sc, t6);
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        Tb[i][j] = (i < dim && j < dim) ? t6[sidx(dim, i, j)] : F(0);
        if (i < dim && j < dim) TbT += Tb[i][j] * Tc[sidx(dim, i, j)];
      }
  }
  const F rcf = narrow<F>(rc);
  F rhobar = F(-2) * TbT / rcf;
  const F irc2 = F(1) / (rcf * rcf);  // one division for the nine components below
  F sigbar[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) sigbar[i][j] = Tb[i][j] * irc2;
  for (int i = 0; i < dim; ++i) trSig += sigbar[i][i];
  // sigma = -p_hat I + (1 - d) S_tilde
  const F phatbar = -trSig;
  const F pbar = p >= F(0) ? phatbar : (F(1) - dd) * phatbar;
  F Stbar[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) Stbar[i][j] = (F(1) - dd) * sigbar[i][j];
  // ---- reverse: dS = 2 mu (eps_dot - tr/D I) + R S_t - S_t R ----
  F Sdb[3][3];  // full-matrix cotangent of dS (symmetric)
  {
    double s64[6];
    F s6[6];
    for (int k = 0; k < 6; ++k) s64[k] = A.bdS && strength && k < ns ? A.bdS[(int64_t)k * A.n + c] : 0.0;
    narrow_n<6>(s64, sc, s6);
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        const F cst = (i < dim && j < dim) ? s6[sidx(dim, i, j)] : F(0);
        Sdb[i][j] = (i == j) ? cst : F(0.5) * cst;
      }
  }
  F ed[3][3], Rr[3][3], tr = F(0);
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      ed[i][j] = F(0.5) * (gv[i][j] + gv[j][i]);
      Rr[i][j] = F(0.5) * (gv[i][j] - gv[j][i]);
    }
  for (int i = 0; i < dim; ++i) tr += ed[i][i];
  F mubar = F(0), trSdb = F(0);
  for (int i = 0; i < dim; ++i) trSdb += Sdb[i][i];
  const F tr_d = tr / F(dim), trSdb_d = trSdb / F(dim);
  for (int i = 0; i < dim; ++i)
    for (int j = 0; j < dim; ++j) mubar += F(2) * (ed[i][j] - (i == j ? tr_d : F(0))) * Sdb[i][j];
  F edbar[3][3], Rbar[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      edbar[i][j] = (i < dim && j < dim) ? F(2) * mu * (Sdb[i][j] - (i == j ? trSdb_d : F(0))) : F(0);
      F a1 = F(0), a2 = F(0), b1 = F(0), b2 = F(0);
      for (int k = 0; k < dim; ++k) {
        a1 += Sdb[i][k] * St[k][j];  // Z S_t
        a2 += St[i][k] * Sdb[k][j];  // S_t Z
        b1 += Rr[i][k] * Sdb[k][j];  // R Z
        b2 += Sdb[i][k] * Rr[k][j];  // Z R
      }
      Rbar[i][j] = (i < dim && j < dim) ? a1 - a2 : F(0);
      if (i < dim && j < dim) Stbar[i][j] += -b1 + b2;
    }
  if (!strength)
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) edbar[i][j] = Rbar[i][j] = F(0);
  F gvbar[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j)
      gvbar[i][j] = F(0.5) * (edbar[i][j] + edbar[j][i]) + F(0.5) * (Rbar[i][j] - Rbar[j][i]);
  // ---- reverse: S_t = f_Y S (stored components) ----
  F Y0bar = F(0);
  if (strength && A.gS) {
    F Stb_st[6], S_st[6];
    for (int i = 0; i < dim; ++i)
      for (int j = i; j < dim; ++j) {
        const int k = sidx(dim, i, j);
        Stb_st[k] = (i == j) ? Stbar[i][i] : Stbar[i][j] + Stbar[j][i];
        S_st[k] = S[i][j];
      }
    F proj = F(0);
    for (int k = 0; k < ns; ++k) proj += Stb_st[k] * S_st[k];
    const bool yielding = M.Y0 > 0.0 && J2 > F(0) && Y0 * Y0 / (F(3) * J2) < F(1);
    const F fjp = yielding ? fY / J2 * proj : F(0);
    for (int k = 0; k < ns; ++k) {
      F sb = Stb_st[k];
      if (yielding) {
        const F wk = k < dim ? F(1) : F(2);
        sb = fY * Stb_st[k] - fjp * wk * S_st[k];
      }
      A.gS[(int64_t)k * A.n + c] += widen(sb, isc);
    }
    if (yielding) Y0bar = proj * F(2) * fY / Y0;
  }
  // ---- reverse: EOS ----
  const F csbar = narrow<F>(A.csbar[c], sc);
  F ubar = pbar * pu;
  rhobar += pbar * pr;
  F Kbar = F(0);
  if constexpr (MIXED) {
    const float Kref = (float)fmax(fmax(M.K0, M.A_T), M.B_T);
    rhobar += csbar * dcr;
    ubar += csbar * dcu;
    if (Kref > 0.f) Kbar = (pbar * dps + csbar * dcs) / Kref;
  } else {
    const double er = 1e-6 * rc, eu = 1e-6 * (fabs(uc) + 1e-3 * fabs(M.E0) + 1e-30), es = 1e-6;
    const double Kref = fmax(fmax(M.K0, M.A_T), M.B_T);
    // the six evaluations of the central differences (rho +-, u +-, scale +-)
    // in one loop, so that the equation of state is emitted once here: six
    // inlined copies overflowed the instruction cache.  c+ + (-c-) from zero is
    // the same value as c+ - c-.
#pragma unroll 1
    for (int k = 0; k < 6; ++k) {
      if (k < 4 ? csbar == 0.0 : !(Kref > 0.0)) continue;
      const double sg = (k & 1) ? -1.0 : 1.0;
      const double r1 = k == 0 ? rc + er : (k == 1 ? rc - er : rc);
      const double u1 = k == 2 ? uc + eu : (k == 3 ? uc - eu : uc);
      const double s1 = k == 4 ? 1.0 + es : (k == 5 ? 1.0 - es : 1.0);
      double p1, c1;
      eos_scaled(M, s1, r1, u1, p1, c1, nullptr, nullptr);
      if (k < 2) {
        dcr += sg * c1;
      } else if (k < 4) {
        dcu += sg * c1;
      } else {
        dps += sg * p1;
        dcs += sg * c1;
      }
    }
    if (csbar != 0.0) {
      rhobar += csbar * dcr / (2.0 * er);
      ubar += csbar * dcu / (2.0 * eu);
    }
    if (Kref > 0.0) Kbar = (pbar * dps + csbar * dcs) / (2.0 * es * Kref);
  }
  // ---- reverse: grad v = G C, C = L^-1 ----
  F Gbar[3][3], Lbar[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      F s = F(0);
      for (int k = 0; k < dim; ++k) s += gvbar[i][k] * C[j][k];  // gvbar C^T
      Gbar[i][j] = (i < dim && j < dim) ? s : F(0);
      Lbar[i][j] = F(0);
    }
  if (corr) {
    F Cbar[3][3], T1[3][3];
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        F s = F(0);
        for (int k = 0; k < dim; ++k) s += G[k][i] * gvbar[k][j];  // G^T gvbar
        Cbar[i][j] = s;
      }
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        F s = F(0);
        for (int k = 0; k < dim; ++k) s += Cbar[i][k] * C[j][k];  // Cbar C^T
        T1[i][j] = s;
      }
    for (int i = 0; i < dim; ++i)
      for (int j = 0; j < dim; ++j) {
        F s = F(0);
        for (int k = 0; k < dim; ++k) s += C[k][i] * T1[k][j];  // C^T (Cbar C^T)
        Lbar[i][j] = -s;
      }
  }
  // ---- reverse: drho = rho * sum_rho ; dx = v + xsph * xs (FP64, unscaled) ----
  const double bdr = A.bdrho ? A.bdrho[c] : 0.0;
  A.grho[c] += widen(rhobar, isc) + bdr * srho;
  A.gu[c] += widen(ubar, isc);
  for (int i = 0; i < dim; ++i)
    if (A.bdx[i]) A.gv[i][c] += A.bdx[i][c];
  if constexpr (MIXED) {
    // the cotangents of the pass-A sums in code units (see ACot): the
    // continuity sum and G are rates (1/T), L is a number, XSPH a velocity
    const Units &U = *A.U;
    float v[24];
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        v[1 + 3 * i + j] = Lbar[i][j];
        v[10 + 3 * i + j] = Gbar[i][j];
      }
    shift_n<9>(v + 1, isc);
    shift_n<9>(v + 10, isc * U.invT);
    v[0] = narrow<float>(rc * bdr, U.invT);
    for (int i = 0; i < 3; ++i) v[19 + i] = (i < dim && A.bdx[i]) ? narrow<float>(P.xsph * A.bdx[i][c], U.V) : 0.f;
    v[22] = v[23] = 0.f;
    for (int q = 0; q < 6; ++q)
      A.Apk[(int64_t)q * ld + c] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
  } else {
    double *I = A.inter;
    I[c] = rc * bdr;
    // the layout of k_adj_passA: L's cotangent enters through d^T Lbar d only
    for (int i = 0; i < dim; ++i)
      for (int j = i; j < dim; ++j)
        I[(1 + sidx(dim, i, j)) * ld + c] = i == j ? (double)Lbar[i][i] : (double)(Lbar[i][j] + Lbar[j][i]);
    for (int i = 0; i < dim; ++i)
      for (int j = 0; j < dim; ++j) I[(7 + 3 * i + j) * ld + c] = Gbar[i][j];
    for (int i = 0; i < dim; ++i) I[(16 + i) * ld + c] = A.bdx[i] ? P.xsph * A.bdx[i][c] : 0.0;
  }
  A.pbar[c] = strength ? widen(mubar, isc) : 0.0;
  A.pbar[ld + c] = widen(Y0bar, isc);
  A.pbar[2 * ld + c] = widen(Kbar, isc);
}

// ---------------------------------------------------------------------------
// Reverse of one pass-A pair term of particle a with partner b:
//   sum_rho += vol_b w.g,  L -= vol_b d (x) g,  G -= vol_b w (x) g,
//   xs -= 2 m_b/(rho_a + rho_b) W w,   vol_b = m_b / rho_b
// ---------------------------------------------------------------------------
// Cotangents of the pass-A sums of one particle: continuity sum, L, G, XSPH.
template <class R>
struct ACot {
  R sr, Lb[3][3], Gb[3][3], xb[3];
};

// K: the kernel factors of the pair, r = |d|; Ct: the cotangents of the sums
// of the particle whose term this is.
template <class R>
__device__ void pairA_adj(int dim, const R d[3], const R w[3], R r, const KPair<R> &K, R mb, R rho_a, R rho_b,
                          const ACot<R> &Ct, R dbar[3], R wbar[3], R &rho_a_bar, R &rho_b_bar) {
  const R vol = mb / rho_b;
  R g[3] = {0, 0, 0};
  for (int i = 0; i < dim; ++i) g[i] = K.phi * d[i];
  const R sr = Ct.sr;
  R gbar[3] = {0, 0, 0}, wg = R(0);
  for (int i = 0; i < 3; ++i) {
    dbar[i] = R(0);
    wbar[i] = R(0);
  }
  for (int i = 0; i < dim; ++i) wg += w[i] * g[i];
  R volbar = sr * wg;
  for (int i = 0; i < dim; ++i) {
    gbar[i] += sr * vol * w[i];
    wbar[i] += sr * vol * g[i];
  }
  // L and G
  for (int i = 0; i < dim; ++i) {
    R Lg = R(0), Gg = R(0), LTd = R(0), GTw = R(0);
    for (int j = 0; j < dim; ++j) {
      Lg += Ct.Lb[i][j] * g[j];
      Gg += Ct.Gb[i][j] * g[j];
      LTd += Ct.Lb[j][i] * d[j];
      GTw += Ct.Gb[j][i] * w[j];
    }
    dbar[i] += -vol * Lg;
    wbar[i] += -vol * Gg;
    gbar[i] += -vol * (LTd + GTw);
    volbar += -d[i] * Lg - w[i] * Gg;
  }
  // XSPH
  rho_a_bar = R(0);
  rho_b_bar = R(0);
  R wx = R(0);
  for (int i = 0; i < dim; ++i) wx += w[i] * Ct.xb[i];
  if (wx != R(0)) {
    const R cc = R(2) * mb / (rho_a + rho_b);
    for (int i = 0; i < dim; ++i) wbar[i] += -cc * K.W * Ct.xb[i];
    const R Wbar = -cc * wx;
    const R ccbar = -K.W * wx;
    const R dcc = -cc / (rho_a + rho_b);
    rho_a_bar += ccbar * dcc;
    rho_b_bar += ccbar * dcc;
    if (r > R(0))
      for (int i = 0; i < dim; ++i) dbar[i] += Wbar * K.phi * d[i];  // dW/dr d / r
  }
  R gd = R(0);
  for (int i = 0; i < dim; ++i) gd += gbar[i] * d[i];
  for (int i = 0; i < dim; ++i) dbar[i] += K.phi * gbar[i] + K.dphi_r * gd * d[i];
  rho_b_bar += -volbar * vol / rho_b;
}

// FP64.  As in pass B both terms of a pair are one form in d and w,
//   phi (alpha w.d - d^T Lam d - w^T Gam d) - W w.xi,
// with alpha = V_e sr_c + V_c sr_e, Lam and Gam the same combinations of the
// cotangents of L (symmetric part) and G, xi = 2 (m_e xb_c - m_c xb_e) / (rho_c +
// rho_e); only the derivative of V_c in rho_c needs e's term by itself.  About
// 180 FP64 instructions a pair instead of 430 (33k particles: 1.23 -> 0.64
// ms).
template <int DIM>
__global__ void k_adj_passA(AdjArgs A) {
  const int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> A.lane_shift;
  if (c >= A.n) return;
  const Lanes64 ln(A.lane_shift);
  constexpr int NS = DIM == 3 ? 6 : 3;
  const int64_t ld = A.ld;
  const double *I = A.inter;
  const bool xsph = A.prm.xsph != 0.0;
  double xc[DIM], vc[DIM], Lc[NS], Gc[DIM][DIM], xb[DIM];
#pragma unroll
  for (int i = 0; i < DIM; ++i) {
    xc[i] = A.x[i][c];
    vc[i] = A.v[i][c];
    xb[i] = I[(16 + i) * ld + c];
#pragma unroll
    for (int j = 0; j < DIM; ++j) Gc[i][j] = I[(7 + 3 * i + j) * ld + c];
  }
#pragma unroll
  for (int q = 0; q < NS; ++q) Lc[q] = I[(1 + q) * ld + c];
  const double src = I[c], rc = A.rho[c], mc = A.m[c], Vc = A.pk.vol[c];
  Support64<DIM> H;
  H.start(A.h[c]);
  double gx[DIM], gv[DIM], gvol = 0.0, gxs = 0.0;
#pragma unroll
  for (int i = 0; i < DIM; ++i) gx[i] = gv[i] = 0.0;
  const int cnt = A.nb_cnt[c];
  for (int k = ln.sub; k < cnt; k += ln.n) {
    const int32_t e = A.nb_idx[(int64_t)k * ld + c];
    const double Ve = A.pk.vol[e];
    double d[DIM], w[DIM], r2 = 0.0, wd = 0.0;
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      d[i] = xc[i] - A.x[i][e];
      w[i] = vc[i] - A.v[i][e];
      r2 = fma(d[i], d[i], r2);
      wd = fma(w[i], d[i], wd);
    }
    H.partner(A.h[e]);
    double phi, dphi, q;
    radial64(H, r2, phi, dphi, q);
    // e's term per unit volume, and the combined coefficients applied to d and w
    const double sre = I[e], al = fma(Ve, src, Vc * sre);
    double te = sre * wd, qd = al * wd;
    double lam[DIM], gam[DIM], gat[DIM];  // (Lam + Lam^T) d, Gam d, Gam^T w
#pragma unroll
    for (int i = 0; i < DIM; ++i) lam[i] = gam[i] = gat[i] = 0.0;
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
      for (int j = i; j < DIM; ++j) {  // row symk: the sum of both off-diagonal entries
        const int s = symk(DIM, i, j);
        const double le = I[(1 + s) * ld + e], l = fma(Ve, Lc[s], Vc * le), dd = d[i] * d[j];
        te = fma(-le, dd, te);
        qd = fma(-l, dd, qd);
        if (i == j) {
          lam[i] = fma(2.0 * l, d[i], lam[i]);
        } else {
          lam[i] = fma(l, d[j], lam[i]);
          lam[j] = fma(l, d[i], lam[j]);
        }
      }
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
      for (int j = 0; j < DIM; ++j) {
        const double ge = I[(7 + 3 * i + j) * ld + e], g = fma(Ve, Gc[i][j], Vc * ge);
        te = fma(-ge, w[i] * d[j], te);
        gam[i] = fma(g, d[j], gam[i]);
        gat[j] = fma(g, w[i], gat[j]);
      }
#pragma unroll
    for (int i = 0; i < DIM; ++i) qd = fma(-w[i], gam[i], qd);
    double cd = dphi * qd;
    if (xsph) {
      const double me = A.m[e], ir = rcp64(rc + A.rho[e]), W = value64(q) * H.hD * (1.0 / 6.0);
      double wx = 0.0;
#pragma unroll
      for (int i = 0; i < DIM; ++i) {
        const double xi = 2.0 * ir * fma(me, xb[i], -mc * I[(16 + i) * ld + e]);
        wx = fma(w[i], xi, wx);
        gv[i] = fma(-W, xi, gv[i]);
      }
      cd = fma(-phi, wx, cd);
      gxs = fma(W * ir, wx, gxs);
    }
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      gx[i] = fma(phi, fma(al, w[i], -lam[i] - gat[i]), fma(cd, d[i], gx[i]));
      gv[i] = fma(phi, fma(al, d[i], -gam[i]), gv[i]);
    }
    gvol = fma(phi, te, gvol);
  }
  const double norm = 6.0 * kernel_sigma<double>(DIM);
  // dV_c / drho_c = -V_c / rho_c
  const double grho = norm * ln.sum(gxs - gvol * (Vc / rc));
#pragma unroll
  for (int i = 0; i < DIM; ++i) {
    gx[i] = norm * ln.sum(gx[i]);
    gv[i] = norm * ln.sum(gv[i]);
  }
  if (ln.sub) return;
#pragma unroll
  for (int i = 0; i < DIM; ++i) {
    A.gx[i][c] += gx[i];
    A.gv[i][c] += gv[i];
  }
  A.grho[c] += grho;
}

// Per-instance, per-material sums of the particle parameter cotangents,
// param_bar[(inst * nmat + mat) * 3 + k], in a fixed order.  Block (inst, j)
// sums the j-th of gy equal chunks of its instance (a strided loop, then a
// tree in shared memory); with part set it stores that partial sum, and
// k_adj_params_final adds the gy partials of each entry.  With
// part NULL (gy = 1) the block adds its instance's sum to out itself.
constexpr int kParamThreads = 256;
constexpr int64_t kParamChunk = 4096;  // particles per block, about
__global__ void __launch_bounds__(kParamThreads) k_adj_params(const double *__restrict__ pbar, int64_t ld,
                                                              const int32_t *__restrict__ mat,
                                                              const int64_t *__restrict__ inst_off, int ninst,
                                                              int64_t n, int nmat, int gy, double *part, double *out) {
  const int inst = blockIdx.x, j = blockIdx.y;
  const int64_t lo0 = (ninst > 1 && inst_off) ? inst_off[inst] : 0;
  const int64_t hi0 = (ninst > 1 && inst_off) ? inst_off[inst + 1] : n;
  const int64_t len = hi0 - lo0, ch = (len + gy - 1) / gy;
  const int64_t lo = lo0 + min(len, (int64_t)j * ch), hi = lo0 + min(len, (int64_t)(j + 1) * ch);
  __shared__ double sh[kParamThreads][3];
  for (int mm = 0; mm < nmat; ++mm) {
    double acc[3] = {0, 0, 0};
    for (int64_t i = lo + threadIdx.x; i < hi; i += kParamThreads) {
      const int mi0 = mat ? mat[i] : 0;
      const int mi = (mi0 >= 0 && mi0 < nmat) ? mi0 : 0;
      if (mi != mm) continue;
      for (int k = 0; k < 3; ++k) acc[k] += pbar[k * ld + i];
    }
    for (int k = 0; k < 3; ++k) sh[threadIdx.x][k] = acc[k];
    __syncthreads();
    for (int s = kParamThreads / 2; s > 0; s >>= 1) {
      if (threadIdx.x < s)
        for (int k = 0; k < 3; ++k) sh[threadIdx.x][k] += sh[threadIdx.x + s][k];
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      const int64_t q = (int64_t)inst * nmat + mm;
      for (int k = 0; k < 3; ++k) {
        if (part) part[(q * gy + j) * 3 + k] = sh[0][k];
        else out[q * 3 + k] += sh[0][k];
      }
    }
    __syncthreads();
  }
}

// A warp per entry: lane i adds the partials i, i + 32, ..., then the lanes in a
// fixed order (a thread per entry, one partial after the other: 23 us at 1M)
__global__ void k_adj_params_final(const double *__restrict__ part, int64_t m, int gy, double *out) {
  const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;  // entry (inst * nmat + mat) * 3 + k
  if (t >= m) return;
  const int lane = threadIdx.x & 31;
  const int64_t q = t / 3;
  const int k = (int)(t - 3 * q);
  double s = 0.0;
  for (int j = lane; j < gy; j += 32) s += part[(q * gy + j) * 3 + k];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) out[t] += s;
}

// The parameter cotangents of all particles (c->ag, 3 x cap_n) summed into
// param_bar; the adjoint's intermediate buffer holds the partial sums (it is
// free once pass A's reverse has read it).
static void adj_params_sum(sph_ctx *c, const int32_t *mat, const int64_t *inst_off, int ninst, int64_t n, int nmat,
                           double *param_bar, cudaStream_t st) {
  int64_t g = (n / ninst + kParamChunk - 1) / kParamChunk;
  int gy = (int)std::max<int64_t>(1, std::min<int64_t>(1024, g));
  if ((int64_t)ninst * nmat * gy * 3 > (int64_t)22 * c->cap_n) gy = 1;
  double *part = gy > 1 ? c->adj_inter : nullptr;
  { k_adj_params<<<dim3(ninst, gy), kParamThreads, 0, st>>>(c->ag, c->cap_n, mat, inst_off, ninst, n, nmat, gy, part,
                                                          param_bar); ++sph::g_launches; }
  if (part) {
    const int64_t m = (int64_t)ninst * nmat * 3;
    { k_adj_params_final<<<nblk(32 * m, 256), 256, 0, st>>>(part, m, gy, param_bar); ++sph::g_launches; }
  }
}

// ---------------------------------------------------------------------------
// Mixed precision (requested precision SPH_MIXED): the pair terms of passes B
// and A are differentiated in FP32, in the code units of the forward
// evaluation (powers of two, so every conversion is exact), on differences of
// the hi/lo-split positions and velocities as in the forward pass, with
// Kahan-compensated FP32 sums.  A quantity q in SI is q_code * U_q, so its
// cotangent in SI is the code-unit cotangent divided by U_q, and a given output
// cotangent enters in code units multiplied by U_q.
// ---------------------------------------------------------------------------
// Output cotangents of dv/dt and du/dt into code units for pass B.
__global__ void k_adj_pack_cot32(AdjArgs A) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= A.n) return;
  const Units &U = *A.U;
  float vb[3] = {0.f, 0.f, 0.f};
  for (int i = 0; i < A.dim; ++i)
    if (A.bdv[i]) vb[i] = narrow<float>(A.bdv[i][c], U.acc);
  const float ub = A.bdu ? narrow<float>(A.bdu[c], U.E * U.invT) : 0.f;
  A.Bpk[c] = make_float4(vb[0], vb[1], vb[2], ub);
}

__device__ __forceinline__ void load_T32(const AdjArgs &A, int64_t b, float t[6], float &cs) {
  const float4 t0 = A.Tf[b], t1 = A.Tf[A.ld + b];
  t[0] = t0.x;
  t[1] = t0.y;
  t[2] = t0.z;
  t[3] = t0.w;
  t[4] = t1.x;
  t[5] = t1.y;
  cs = t1.z;
}

template <int DIM>
__global__ void k_adj_passB32(AdjArgs A) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= A.n) return;
  constexpr int dim = DIM;
  const int ns = nsym(dim);
  const float4 Pc = A.pk.px(c), Qc = A.pk.pxl(c), Vc = A.pk.pv(c), Wc = A.pk.pvl(c);
  float Tc[6], csc;
  load_T32(A, c, Tc, csc);
  const float4 bc = A.Bpk[c];
  const float vbc[3] = {bc.x, bc.y, bc.z};
  KahanT<float> gx[3], gv[3], Tb[6], csb, rhb;
  const int cnt = A.nb_cnt[c];
  AdjCursor cur;
  cur.start(A, c, cnt);
  for (int k = 0; k < cnt; ++k) {
    float4 Pe, Qe;
    const int32_t e = cur.next(A, k, Pe, Qe);
    const float4 Ve = A.pk.pv(e), We = A.pk.pvl(e);
    float d[3] = {(Pc.x - Pe.x) + (Qc.x - Qe.x), (Pc.y - Pe.y) + (Qc.y - Qe.y),
                  DIM == 3 ? (Pc.z - Pe.z) + (Qc.z - Qe.z) : 0.f};
    float w[3] = {(Vc.x - Ve.x) + (Wc.x - We.x), (Vc.y - Ve.y) + (Wc.y - We.y),
                  DIM == 3 ? (Vc.z - Ve.z) + (Wc.z - We.z) : 0.f};
    float Te[6], cse;
    load_T32(A, e, Te, cse);
    const float4 be = A.Bpk[e];
    const float vbe[3] = {be.x, be.y, be.z};
    const float hab = 0.5f * (Pc.w + Pe.w);
    float r2 = 0.f;
    for (int i = 0; i < dim; ++i) r2 += d[i] * d[i];
    const KPair<float> K = kernel_pair<float>(dim, sqrtf(r2), hab);
    const VPair<float> Vs = visc_pair<float>(dim, d, w, r2, hab, Vc.w, Ve.w, csc, cse, A.f_alpha, A.f_beta, A.f_eps_v);
    float db[3], wb[3], Bs[6], csh, rh;
    pairB_adj<float>(dim, d, w, K, Vs, Tc, Te, Qe.w, vbc, bc.w, db, wb, Bs, csh, rh);  // c's own term
    for (int i = 0; i < dim; ++i) {
      gx[i].add(db[i]);
      gv[i].add(wb[i]);
    }
    for (int q = 0; q < ns; ++q) Tb[q].add(Bs[q]);
    csb.add(csh);
    rhb.add(rh);
    const float dn[3] = {-d[0], -d[1], -d[2]}, wn[3] = {-w[0], -w[1], -w[2]};
    pairB_adj<float>(dim, dn, wn, K, Vs, Te, Tc, Qc.w, vbe, be.w, db, wb, Bs, csh, rh);  // e's term, w.r.t. c
    for (int i = 0; i < dim; ++i) {
      gx[i].add(-db[i]);
      gv[i].add(-wb[i]);
    }
    for (int q = 0; q < ns; ++q) Tb[q].add(Bs[q]);
    csb.add(csh);
    rhb.add(rh);
  }
  const Units &U = *A.U;
  for (int i = 0; i < dim; ++i) {
    A.gx[i][c] += gx[i].value() * U.invL;
    A.gv[i][c] += gv[i].value() * U.invV;
  }
  A.grho[c] += rhb.value() * U.invrho;
  const double uTinv = U.rho * U.rho * U.invsig;
  for (int q = 0; q < 6; ++q) A.Tbar[(int64_t)q * A.ld + c] = q < ns ? Tb[q].value() * uTinv : 0.0;
  A.csbar[c] = csb.value() * U.invV;
}

__device__ __forceinline__ ACot<float> load_acot32(const AdjArgs &A, int64_t a) {
  float v[24];
  for (int q = 0; q < 6; ++q) {
    const float4 t = A.Apk[(int64_t)q * A.ld + a];
    v[4 * q] = t.x;
    v[4 * q + 1] = t.y;
    v[4 * q + 2] = t.z;
    v[4 * q + 3] = t.w;
  }
  ACot<float> c;
  c.sr = v[0];
  for (int i = 0; i < 3; ++i) {
    for (int j = 0; j < 3; ++j) {
      c.Lb[i][j] = v[1 + 3 * i + j];
      c.Gb[i][j] = v[10 + 3 * i + j];
    }
    c.xb[i] = v[19 + i];
  }
  return c;
}

template <int DIM>
__global__ void k_adj_passA32(AdjArgs A) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= A.n) return;
  constexpr int dim = DIM;
  const float4 Pc = A.pk.px(c), Qc = A.pk.pxl(c), Vc = A.pk.pv(c), Wc = A.pk.pvl(c);
  const ACot<float> Cc = load_acot32(A, c);
  KahanT<float> gx[3], gv[3], grho;
  const int cnt = A.nb_cnt[c];
  AdjCursor cur;
  cur.start(A, c, cnt);
  for (int k = 0; k < cnt; ++k) {
    float4 Pe, Qe;
    const int32_t e = cur.next(A, k, Pe, Qe);
    const float4 Ve = A.pk.pv(e), We = A.pk.pvl(e);
    float d[3] = {(Pc.x - Pe.x) + (Qc.x - Qe.x), (Pc.y - Pe.y) + (Qc.y - Qe.y),
                  DIM == 3 ? (Pc.z - Pe.z) + (Qc.z - Qe.z) : 0.f};
    float w[3] = {(Vc.x - Ve.x) + (Wc.x - We.x), (Vc.y - Ve.y) + (Wc.y - We.y),
                  DIM == 3 ? (Vc.z - Ve.z) + (Wc.z - We.z) : 0.f};
    const float hab = 0.5f * (Pc.w + Pe.w);
    float r2 = 0.f;
    for (int i = 0; i < dim; ++i) r2 += d[i] * d[i];
    const float r = sqrtf(r2);
    const KPair<float> K = kernel_pair<float>(dim, r, hab);
    float db[3], wb[3], ra, rb;
    pairA_adj<float>(dim, d, w, r, K, Qe.w, Vc.w, Ve.w, Cc, db, wb, ra, rb);  // c's own term
    for (int i = 0; i < dim; ++i) {
      gx[i].add(db[i]);
      gv[i].add(wb[i]);
    }
    grho.add(ra);
    const ACot<float> Ce = load_acot32(A, e);
    const float dn[3] = {-d[0], -d[1], -d[2]}, wn[3] = {-w[0], -w[1], -w[2]};
    pairA_adj<float>(dim, dn, wn, r, K, Qc.w, Ve.w, Vc.w, Ce, db, wb, ra, rb);  // e's term, w.r.t. c
    for (int i = 0; i < dim; ++i) {
      gx[i].add(-db[i]);
      gv[i].add(-wb[i]);
    }
    grho.add(rb);
  }
  const Units &U = *A.U;
  for (int i = 0; i < dim; ++i) {
    A.gx[i][c] += gx[i].value() * U.invL;
    A.gv[i][c] += gv[i].value() * U.invV;
  }
  A.grho[c] += grho.value() * U.invrho;
}

void rhs_adjoint(sph_ctx *c, const sph_state *s, const MatTable &mt, const sph_params &p, const sph_derivs &dbar,
                 sph_state *sbar, double *param_bar, cudaStream_t st) {
  const int64_t n = s->n;
  if (n == 0) return;
  AdjArgs A;
  memset(&A, 0, sizeof(A));
  A.dim = s->dim;
  A.n = n;
  A.ld = c->cap_n;
  for (int k = 0; k < 3; ++k) {
    A.x[k] = s->x[k];
    A.v[k] = s->v[k];
    A.bdx[k] = dbar.dx[k];
    A.bdv[k] = dbar.dv[k];
    A.gx[k] = sbar->x[k];
    A.gv[k] = sbar->v[k];
  }
  A.rho = s->rho;
  A.u = s->u;
  A.m = s->m;
  A.h = s->h;
  A.S = s->S;
  A.dmg = s->dmg;
  A.mat = s->mat;
  A.nb_idx = c->nb_idx;
  A.nb_cnt = c->nb_cnt;
  A.T = (const double *)c->T;
  A.cs = c->cs;
  A.bdrho = dbar.drho;
  A.bdu = dbar.du;
  A.bdS = dbar.dS;
  A.grho = sbar->rho;
  A.gu = sbar->u;
  A.gS = sbar->S;
  // scratch: the step buffers of the second derivative set are free here
  A.Tbar = c->st.d_S[1];
  A.csbar = c->st.d_cs[1];
  A.inter = c->adj_inter;
  A.pbar = c->ag;
  A.mt = mt;
  A.prm = p;
  const int T = 128;
  if (p.precision == SPH_MIXED) {
    A.pk = c->pk;
    A.Tf = (const float4 *)c->T;
    A.Bpk = c->adj32;
    A.Apk = c->adj32 + c->cap_n;
    A.U = c->units;
    A.sums = c->adj_sums;
    A.f_alpha = (float)p.alpha;
    A.f_beta = (float)p.beta;
    A.f_eps_v = (float)p.eps_v;
    { k_adj_pack_cot32<<<nblk(n, 256), 256, 0, st>>>(A); ++sph::g_launches; }
    if (s->dim == 3) {
      { k_adj_passB32<3><<<nblk(n, T), T, 0, st>>>(A); ++sph::g_launches; }
      { k_adj_update<true, 3><<<nblk(n, T), T, 0, st>>>(A); ++sph::g_launches; }
    } else {
      { k_adj_passB32<2><<<nblk(n, T), T, 0, st>>>(A); ++sph::g_launches; }
      { k_adj_update<true, 2><<<nblk(n, T), T, 0, st>>>(A); ++sph::g_launches; }
    }
    if (s->dim == 3) { k_adj_passA32<3><<<nblk(n, T), T, 0, st>>>(A); ++sph::g_launches; }
    else { k_adj_passA32<2><<<nblk(n, T), T, 0, st>>>(A); ++sph::g_launches; }
  } else {
    A.pk = c->pk;
    A.lane_shift = lanes64_shift(n, c->num_sms);
    const int T64 = threads64(n, c->num_sms, T), g = nblk(n << A.lane_shift, T64), gu = nblk(n, T64);
    if (s->dim == 3) {
      k_adj_passB<3><<<g, T64, 0, st>>>(A);
      k_adj_update<false, 3><<<gu, T64, 0, st>>>(A);
      k_adj_passA<3><<<g, T64, 0, st>>>(A);
    } else {
      k_adj_passB<2><<<g, T64, 0, st>>>(A);
      k_adj_update<false, 2><<<gu, T64, 0, st>>>(A);
      k_adj_passA<2><<<g, T64, 0, st>>>(A);
    }
    sph::g_launches += 3;
  }
  const int ninst = s->ninst > 0 ? s->ninst : 1;
  if (param_bar) adj_params_sum(c, s->mat, s->inst_off, ninst, n, mt.nmat, param_bar, st);
}

// ---------------------------------------------------------------------------
// Reverse of out = Y(base + frac dt d): the state cotangent passes to base,
// frac dt times it to the derivatives, through the yield map for S.
// ---------------------------------------------------------------------------
struct PcAdjArgs {
  int dim;
  int64_t n;
  const double *bS, *dS;
  const int32_t *mat;
  const int64_t *inst_off;
  int ninst;
  const double *dt;
  double frac;
  MatTable mt;
  const double *ox[3], *ov[3], *orho, *ou, *oS;   // cotangent of out
  double *gx[3], *gv[3], *grho, *gu, *gS;         // base cotangent (+=)
  double *fx[3], *fv[3], *frho, *fu, *fS;         // derivative cotangent (=)
  double *pY;                                     // per-particle Y0 cotangent (=)
  int density_sum;
};

__global__ void k_pc_adj(PcAdjArgs A) {
  const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= A.n) return;
  const int inst = inst_of(A.inst_off, A.ninst, a);
  const double h = A.frac * A.dt[inst];
  for (int ax = 0; ax < A.dim; ++ax) {
    const double lx = A.ox[ax][a], lv = A.ov[ax][a];
    A.gx[ax][a] += lx;
    A.gv[ax][a] += lv;
    A.fx[ax][a] = h * lx;
    A.fv[ax][a] = h * lv;
  }
  A.grho[a] += A.orho[a];
  A.frho[a] = A.density_sum ? 0.0 : h * A.orho[a];
  A.gu[a] += A.ou[a];
  A.fu[a] = h * A.ou[a];
  double yb = 0.0;
  if (A.bS) {
    const int ns = nsym(A.dim);
    const int mi0 = A.mat ? A.mat[a] : 0;
    const sph_material &M = A.mt.m[(mi0 >= 0 && mi0 < A.mt.nmat) ? mi0 : 0];
    double Sp[6], lo[6], J2 = 0.0, proj = 0.0;
    for (int k = 0; k < ns; ++k) {
      Sp[k] = A.bS[(int64_t)k * A.n + a] + h * A.dS[(int64_t)k * A.n + a];
      lo[k] = A.oS[(int64_t)k * A.n + a];
      J2 += (k < A.dim ? 1.0 : 2.0) * Sp[k] * Sp[k];
      proj += lo[k] * Sp[k];
    }
    J2 *= 0.5;
    const bool yielding = M.strength && M.Y0 > 0.0 && J2 > 0.0 && M.Y0 * M.Y0 / (3.0 * J2) < 1.0;
    const double f = yielding ? M.Y0 * M.Y0 / (3.0 * J2) : 1.0;
    for (int k = 0; k < ns; ++k) {
      double sb = lo[k];
      if (yielding) sb = f * lo[k] - f / J2 * proj * (k < A.dim ? 1.0 : 2.0) * Sp[k];
      A.gS[(int64_t)k * A.n + a] += sb;
      A.fS[(int64_t)k * A.n + a] = h * sb;
    }
    if (yielding) yb = proj * 2.0 * f / M.Y0;
  }
  A.pY[a] = yb;
}

void pc_update_adjoint(sph_ctx *c, const sph_state *base, const sph_derivs &d, const double *dt, double frac,
                       const MatTable &mt, const sph_params &p, const sph_state *obar, sph_state *gbar,
                       sph_derivs *fbar, double *param_bar, cudaStream_t st) {
  const int64_t n = base->n;
  if (n == 0) return;
  PcAdjArgs A;
  memset(&A, 0, sizeof(A));
  A.dim = base->dim;
  A.n = n;
  A.bS = base->S;
  A.dS = d.dS;
  A.mat = base->mat;
  A.inst_off = base->inst_off;
  A.ninst = base->ninst > 0 ? base->ninst : 1;
  A.dt = dt;
  A.frac = frac;
  A.mt = mt;
  for (int k = 0; k < 3; ++k) {
    A.ox[k] = obar->x[k];
    A.ov[k] = obar->v[k];
    A.gx[k] = gbar->x[k];
    A.gv[k] = gbar->v[k];
    A.fx[k] = fbar->dx[k];
    A.fv[k] = fbar->dv[k];
  }
  A.orho = obar->rho;
  A.ou = obar->u;
  A.oS = obar->S;
  A.grho = gbar->rho;
  A.gu = gbar->u;
  A.gS = gbar->S;
  A.frho = fbar->drho;
  A.fu = fbar->du;
  A.fS = fbar->dS;
  // per-particle Y0 cotangent in the parameter scratch (mu and K stay zero)
  cudaMemsetAsync(c->ag, 0, sizeof(double) * 3 * c->cap_n, st);
  A.pY = c->ag + c->cap_n;
  A.density_sum = p.density_sum;
  { k_pc_adj<<<nblk(n, 256), 256, 0, st>>>(A); ++sph::g_launches; }
  const int ninst = base->ninst > 0 ? base->ninst : 1;
  if (param_bar) adj_params_sum(c, base->mat, base->inst_off, ninst, n, mt.nmat, param_bar, st);
}

}  // namespace sph
