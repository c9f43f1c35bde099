// FP64 pair arithmetic shared by the neighbour passes and their adjoint.
#pragma once

#include "fp64fast.cuh"
#include "fpbits.cuh"
#include "sph_internal.cuh"

namespace sph {

// ---------------------------------------------------------------------------
// FP64 pair sums.  Bound by the FP64 unit, so each pair is written in as few
// FP64 instructions as its terms need: reciprocals from fp64fast.cuh, V_b read
// from an array (one gather instead of a division), powers of 1/h_ab kept
// while h_b stays the same from partner to partner (a bit test), the kernel
// slope as one product of two linear factors whose coefficients are selected
// by the branch, and the kernel norm applied to the sums.
// ---------------------------------------------------------------------------
template <int DIM>
struct Support64 {
  double ha, hab, hinv, hD, hD1;  // h_a, h_ab, 1/h_ab, its powers D and D + 1
  uint64_t last;                  // bits of the h_b these belong to
  __device__ __forceinline__ void set(double hb) {
    last = dbits(hb);
    hab = 0.5 * (ha + hb);
    hinv = rcp64(hab);
    const double i2 = hinv * hinv;
    hD = DIM == 3 ? i2 * hinv : i2;
    hD1 = hD * hinv;
  }
  __device__ __forceinline__ void start(double h) {
    ha = h;
    set(h);
  }
  __device__ __forceinline__ void partner(double hb) {
    if (dbits(hb) != last) set(hb);
  }
};

// The lanes that share one particle's list: lane `sub` of n takes partners
// sub, sub + n, ...  Sums are combined over the group in a fixed order.
struct Lanes64 {
  int sub, n;
  unsigned mask;
  __device__ __forceinline__ Lanes64(int shift) {
    n = 1 << shift;
    const int lane = threadIdx.x & 31;
    sub = lane & (n - 1);
    mask = ((1u << n) - 1u) << (lane - sub);  // n <= 8
  }
  __device__ __forceinline__ double sum(double v) const {
    for (int o = 1; o < n; o <<= 1) v += __shfl_xor_sync(mask, v, o);
    return v;
  }
};

// q < 1/2 for q >= 0, from the bits
__device__ __forceinline__ bool below_half(double q) { return __double2hiint(q) < 0x3fe00000; }

// (h^(D+1) / 6 sigma) dW/dr at q = r/h: q (3q - 2), or -(1 - q)^2 from q = 1/2
__device__ __forceinline__ double slope64(double q) {
  const bool in = below_half(q);
  const double a1 = in ? 1.0 : -1.0, b1 = in ? 0.0 : 1.0, c1 = in ? 3.0 : 1.0, d1 = in ? -2.0 : -1.0;
  return fma(a1, q, b1) * fma(c1, q, d1);
}
// (h^D / sigma) W: 1 + 6 q^2 (q - 1), or 2 (1 - q)^3.  The q of a partner (r^2 <
// h^2) may round above 1, where W is 0: a negative value would give NaN under a
// non-integer power (artificial stress).  The sign of 1 - q is tested on its bits.
__device__ __forceinline__ double value64(double q) {
  const double e = 1.0 - q, t = below_half(q) ? q : ((int64_t)dbits(e) < 0 ? 0.0 : e), t2 = t * t;
  return below_half(q) ? fma(6.0 * t2, t - 1.0, 1.0) : 2.0 * t2 * t;
}

// out = (symmetric components t) g
template <class R>
__device__ __forceinline__ void sym_mv(int dim, const R t[6], const R g[3], R out[3]) {
  if (dim == 3) {
    out[0] = t[0] * g[0] + t[3] * g[1] + t[4] * g[2];
    out[1] = t[3] * g[0] + t[1] * g[1] + t[5] * g[2];
    out[2] = t[4] * g[0] + t[5] * g[1] + t[2] * g[2];
  } else {
    out[0] = t[0] * g[0] + t[2] * g[1];
    out[1] = t[2] * g[0] + t[1] * g[1];
    out[2] = R(0);
  }
}

// phi = (dW/dr) / r and phi'(r) / r in units of 6 sigma, and q; the limits at
// r = 0 are -2 / h^(D+2) and 0.
template <int DIM>
__device__ __forceinline__ void radial64(const Support64<DIM> &H, double r2, double &phi, double &dphi, double &q) {
  const double rinv = rsqrt64(r2);
  q = r2 * rinv * H.hinv;
  const bool in = below_half(q);
  const double s2 = fma(in ? 6.0 : -2.0, q, in ? -2.0 : 2.0) * (H.hD1 * H.hinv);  // second derivative
  phi = slope64(q) * H.hD1 * rinv;
  dphi = (s2 - phi) * (rinv * rinv);
  if (rinv == 0.0) {
    phi = -2.0 * H.hD1 * H.hinv;
    dphi = 0.0;
  }
}

// Launch of an FP64 pair kernel over n particles: lanes per particle (as a
// shift) and threads per block.  What counts is that the warps spread evenly
// over the SMs' FP64 units: one-warp blocks while that leaves fewer than eight
// 128-thread blocks per SM; and with fewer than kLaneWarps warps per SM even
// that leaves the unit idle between dependent operations, so 2, 4 or 8 lanes
// share a particle's list.  After the sums only the first lane of each group goes
// on to the particle's own update, which a warp then runs with 4 to 16 lanes
// active; the measured thresholds include that.
// Against one lane, at thresholds of 2, 4 and 8 warps: rings at 4.4k (ten
// steps) 6.90 -> 5.67, 5.79, 5.80 ms; a right-hand side at 8k 902 -> 815, 804,
// 920 us and at 27k 1078 -> 1080, 1078, 1125 us; RK3 at 14k 3.18 -> 3.18, 2.96,
// 3.25 ms.
constexpr int kLaneWarps = 4;
inline int lanes64_shift(int64_t n, int num_sms) {
  int s = 0;
  while (s < 3 && (n << s) < (int64_t)32 * kLaneWarps * num_sms) ++s;
  return s;
}
inline int threads64(int64_t n, int num_sms, int large) { return nblk(n, 128) < 8 * num_sms ? 32 : large; }

}  // namespace sph
