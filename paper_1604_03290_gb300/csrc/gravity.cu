// Barnes-Hut self-gravity (Sect. 3.3), GB300 form.
//
// A warp walks the pre-order tree for 32 consecutive sorted particles.
// Acceptance stays per particle, exactly as in a per-particle walk: a lane
// that uses node n as a pseudo-particle ignores the rest of n's subtree
// (ids below skip[n]); the warp enters n's children if any lane rejected
// n.  Leaves rejected by a lane are summed particle by particle (self
// skipped), staged through shared memory.  The accepted set of every
// particle - hence the sum - is the one of the per-particle definition:
//   node used iff its cube does not contain a and s / r < theta
//   (s = s0 / 2^level, r = |x_a - com|, evaluated as s < theta * r);
//   a_a = -G sum m_p (x_a - x_p) / (r^2 + eps_a^2)^1.5, eps_a = eps_grav h_a
// (the paper's Eq. gravitational_force read as attractive, with Plummer
// softening).
//
// Reused tree (gravity/hydro decoupling, Sect. 6.3): the pseudo-particles,
// node cubes and leaf membership are those of the build, the particle's cell
// is recomputed from its current position in the build's root cube, and
// leaves are summed at the members' current positions (the packed views are
// refreshed before the walk).
//
// Mixed precision: distances from hi/lo split coordinates in FP32, the
// acceptance test in FP32 with a relative band of 1e-4 around the threshold
// inside which the FP64 expression decides, FP32 monopole terms summed with
// Kahan compensation.
#include "fp64fast.cuh"
#include "morton.cuh"
#include "sph_internal.cuh"

namespace sph {

// One warp (one particle group at a time) per block, 32 resident blocks per
// SM at 64 registers: measured on GB300 (2M cloud) 33.1 ms per step against
// 34.5 (4 warps x 8 blocks), 34.8 (8 x 4) and 36.1 (2 x 16).
#ifndef SPH_GRAV_WARPS
#define SPH_GRAV_WARPS 1
#endif
constexpr int kGrWarps = SPH_GRAV_WARPS;  // warps (particle groups) per block
// resident blocks per SM the walk is compiled for (register budget)
#ifndef SPH_GRAV_MIN_BLOCKS
#define SPH_GRAV_MIN_BLOCKS 32
#endif
// FP64 walk: resident one-warp blocks per SM (80 registers, 8 KB of lists each)
constexpr int kGrav64Blocks = 24;
constexpr float kMacBand = 1e-4f;
constexpr int kFlushTerms = 16;
// A leaf summed directly by few lanes: rather than each of them looping over
// the members while the others wait, the warp takes the lanes one at a time,
// every member lane evaluates its term for that lane, and a butterfly sum
// over the warp gives the leaf's contribution (mixed precision).  Chosen when
// (lanes summing the leaf) x kTransposedCost < (members) x kSerialCost, the
// instruction counts of the two forms per lane and per member.
constexpr int kTransposedCost = 66, kSerialCost = 29;

// Sum of the FP32 terms of one particle: a plain partial sum, added into a
// compensated (Kahan) sum every kFlushTerms terms, so that the error stays
// near that of a compensated sum (the partial sums are short) at a fraction
// of its cost per term.
struct GravSumF {
  float px = 0.f, py = 0.f, pz = 0.f;
  int n = 0;
  KahanT<float> kx, ky, kz;
  __device__ __forceinline__ void flush() {
    kx.add(px);
    ky.add(py);
    kz.add(pz);
    px = py = pz = 0.f;
    n = 0;
  }
  __device__ __forceinline__ void add(float fx, float fy, float fz) {
    px += fx;
    py += fy;
    pz += fz;
    if (++n == kFlushTerms) flush();
  }
  // the term g d; the fused form is written out, so that every instance of the walk rounds alike
  __device__ __forceinline__ void add_scaled(float g, const float d[3]) {
    px = __fmaf_rn(g, d[0], px);
    py = __fmaf_rn(g, d[1], py);
    pz = __fmaf_rn(g, d[2], pz);
    if (++n == kFlushTerms) flush();
  }
  __device__ __forceinline__ void value(double &x, double &y, double &z) {
    flush();
    x = kx.value();
    y = ky.value();
    z = kz.value();
  }
};

// x^2 + y^2 + z^2, its fused operations written out as well
__device__ __forceinline__ float norm2(float x, float y, float z) {
  return __fmaf_rn(z, z, __fmaf_rn(x, x, __fmul_rn(y, y)));
}

// 1 / q^(3/2) from the reciprocal square root in FP32 (a few ulps, far below
// the mixed form's tolerance)
__device__ __forceinline__ float inv_q32(float q) {
  const float r = rsqrtf(q);
  return r * r * r;
}

struct GravArgs {
  Tree T;
  PackedF32 pk;
  const double *x[3], *m, *h;
  int dim;
  double G, theta, eps;
  double *out[3];
  const Units *U;
  int32_t *err;
  int share;  // FP64: 2^share lanes per particle
  // A node whose cube holds the particle also holds its centre of mass, so r <=
  // sqrt(D) s there; with D theta^2 < 1 (by a margin far above the rounding of
  // either test) the opening criterion already rejects it and the containment
  // test can be skipped: the accepted set is the same.  Decided on the host:
  // formed in the kernel, the compiler evaluated the comparison again at every
  // visit (an FP64 instruction each, 37 % of the FP64 unit).
  int test_inside;
  int reuse;  // the tree was built at earlier positions: locate each particle anew
  unsigned long long *ctr;  // NULL, or the interaction counters
};

template <int DIM>
__device__ __forceinline__ double r2_fp64(const double xa[3], double cx, double cy, double cz) {
  double dx = __dsub_rn(xa[0], cx);
  double dy = __dsub_rn(xa[1], cy);
  double r2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
  if (DIM == 3) {
    double dz = __dsub_rn(xa[2], cz);
    r2 = __dadd_rn(r2, __dmul_rn(dz, dz));
  }
  return r2;
}

// Mixed precision.  PACKED (Tree::packed_walk): a node's skip, level and leaf
// flag come from the w word of its second COM view, so that a visit loads two float4
// (the node's member range only when some lane sums it directly), and the
// node edge s0 / 2^level is the instance's FP32 edge shifted by the level:
// the same value k_node_finish stores otherwise.
// INSIDE, COUNT: with the containment test, with the interaction counters.  Each
// costs a few instructions and registers at every visit, so the packed form
// has instances without them: 2M cloud step (neither) 34.1 -> 33.0 ms, 400k pair
// window (containment only) 19.3 -> 18.7 ms, 1 % of it from leaving the warp's
// second vote out at inner nodes.
template <int DIM, bool PACKED, bool INSIDE, bool COUNT>
__global__ void __launch_bounds__(kGrWarps * 32, SPH_GRAV_MIN_BLOCKS) k_gravity(GravArgs A) {
  using R = float;
  __shared__ float4 sh_hi[kGrWarps][kMaxLeaf];  // (x_hi, y_hi, z_hi, G m_b) of leaf members
  __shared__ float4 sh_lo[kGrWarps][kMaxLeaf];
  const Tree &T = A.T;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Warps take groups of particles; acceptance is per particle, so any
  // grouping gives the same sums.  One instance: full chunks of 32
  // consecutive slots (Morton order keeps them close); several: the tree's
  // groups, which never span instances.
  const bool chunks = T.ninst <= 1;
  const int ngroups = chunks ? (int)((T.n + 31) >> 5) : *T.ngroups;
  constexpr int dim = DIM;
  const int L = T.leaf_size, B = T.max_depth;
  const int nnodes = T.iter_cap > 0 ? min(*T.nnodes, T.iter_cap) : *T.nnodes;
  const int64_t cap = T.cap_nodes;
  const double Gs = A.G * A.U->M * A.U->T * A.U->T * A.U->invL * A.U->invL * A.U->invL;
  const R G = (R)Gs;
  for (int g = blockIdx.x * kGrWarps + w; g < ngroups; g += gridDim.x * kGrWarps) {
    const int32_t s0 = chunks ? g * 32 : T.grp_start[g];
    const int32_t s1 = chunks ? (int32_t)(((int64_t)s0 + 32 < T.n) ? (int64_t)s0 + 32 : T.n) : T.grp_end[g];
    const int inst = chunks ? 0 : T.grp_inst[g];
    const int32_t slot = s0 + lane;
    const bool act = slot < s1;
    const int32_t a = act ? (T.perm_identity ? slot : T.perm[slot]) : 0;  // identity: state in tree order
    // the cell of the particle's current position (the key of the build
    // unless the tree is reused); node cubes are those of the build
    double xa[3] = {0, 0, 0};
    if (INSIDE && act)
      for (int ax = 0; ax < dim; ++ax) xa[ax] = A.x[ax][a];
    const unsigned long long ka =
        !INSIDE || !act ? 0ULL
             : (A.reuse ? morton_key(xa, dim, B, inst, T.inst_lo, T.inst_s0[inst], T.inst_rs0[inst]) : T.skey[slot]);
    const float4 Pa = A.pk.px(a), Qa = A.pk.pxl(a);
    const double e = A.eps * (double)Pa.w;
    const R eps2 = (R)(e * e);
    const double s0r = T.inst_s0[inst];
    // the instance's root edge in FP32 code units (PACKED: shifted by the level per node)
    const float s0f = PACKED ? to_f32_scaled(s0r, pow2_exp(A.U->invL), A.U->invL) : 0.f;
    const double th = A.theta;
    const float th2f = (float)(th * th);
    GravSumF acc;
    int32_t skip_until = act ? -1 : 0x7fffffff;  // an idle lane meets no node
    const int32_t root = T.inst_root[inst];
    const int32_t stop = root >= 0 ? T.skip[root] : root;
    int iter = 0;
    unsigned nacc = 0, nterm = 0;  // this lane's accepted nodes and particle terms (counters)
    for (int32_t nd = root; nd < stop && iter <= nnodes; ++iter) {
      int32_t f = 0, e1 = 0, sk;
      int lev;
      bool leaf;
      float4 ch, cl;
      if constexpr (PACKED) {
        ch = T.fcom_hi[nd];
        cl = T.fcom_lo[nd];
        const uint32_t wd = __float_as_uint(cl.w);
        sk = (int32_t)(wd & (uint32_t)kPackedSkip);
        lev = (int)((wd >> 26) & 31u);
        leaf = (wd >> 31) != 0u;
      } else {
        const int4 rec = T.nrec[nd];  // (first, end, skip, level)
        f = rec.x;
        e1 = rec.y;
        sk = rec.z;
        lev = rec.w;
        leaf = (e1 - f <= L) || lev == B;
      }
      bool open = false, direct = false;
      if (nd >= skip_until) {
        const bool inside = INSIDE && A.test_inside && (ka >> (dim * (B - lev))) == T.cell[nd];
        bool accept = false;
        float mpf = 0.f;
        R d[3] = {R(0), R(0), R(0)}, r2 = R(0);
        if (!inside) {
          if constexpr (!PACKED) {
            ch = T.fcom_hi[nd];
            cl = T.fcom_lo[nd];
          }
          d[0] = (Pa.x - ch.x) + (Qa.x - cl.x);
          d[1] = (Pa.y - ch.y) + (Qa.y - cl.y);
          d[2] = (Pa.z - ch.z) + (Qa.z - cl.z);
          r2 = norm2(d[0], d[1], d[2]);
          mpf = ch.w;
          const float sf = PACKED ? __int_as_float(__float_as_int(s0f) - (lev << 23)) : cl.w;
          const float lhs = sf * sf, rhs = th2f * r2;
          if (lhs < rhs * (1.0f - kMacBand)) accept = true;
          else if (lhs > rhs * (1.0f + kMacBand)) accept = false;
          else {
            // rare: the FP64 decision, from values reloaded here rather than kept live in the loop
            const double xr[3] = {A.x[0][a], A.x[1][a], DIM == 3 ? A.x[2][a] : 0.0};
            accept = ldexp(T.inst_s0[inst], -lev) <
                     A.theta * sqrt(r2_fp64<DIM>(xr, T.com[nd], T.com[cap + nd], DIM == 3 ? T.com[2 * cap + nd] : 0.0));
          }
        }
        if (accept) {
          const R mp = mpf;
          const R gq = -G * mp * inv_q32(r2 + eps2);
          acc.add_scaled(gq, d);
          skip_until = sk;
          if constexpr (COUNT) ++nacc;
        } else if (leaf) {
          direct = true;
          skip_until = sk;
        } else {
          open = true;
        }
      }
      if (!leaf) {  // no lane sums it directly
        nd = __any_sync(0xffffffffu, open) ? nd + 1 : sk;
        continue;
      }
      const unsigned dmask = __ballot_sync(0xffffffffu, direct);
      const int32_t node = nd;
      nd = sk;
      if (dmask) {
        if constexpr (PACKED) {
          const int4 rec = T.nrec[node];
          f = rec.x;
          e1 = rec.y;
        }
        for (int32_t base = f; base < e1; base += kMaxLeaf) {
          const int c = min(e1 - base, kMaxLeaf);
          int32_t bm = -1;
          float4 pb = make_float4(0.f, 0.f, 0.f, 0.f), qb = pb;
          if (lane < c) {
            bm = T.perm_identity ? base + lane : T.perm[base + lane];
            pb = A.pk.px(bm);
            qb = A.pk.pxl(bm);
            sh_hi[w][lane] = make_float4(pb.x, pb.y, pb.z, -(float)G * qb.w);  // qb.w = m as float
            sh_lo[w][lane] = make_float4(qb.x, qb.y, qb.z, qb.w);
          }
          __syncwarp();
          const bool transposed = __popc(dmask) * kTransposedCost < c * kSerialCost;
          if (transposed) {
            const float gmk = -(float)G * qb.w;
            unsigned mm = dmask;
            while (mm) {
              const int i = __ffs(mm) - 1;
              mm &= mm - 1;
              // lane i's particle, against member `lane`
              const float ax = __shfl_sync(0xffffffffu, Pa.x, i), ay = __shfl_sync(0xffffffffu, Pa.y, i),
                          az = __shfl_sync(0xffffffffu, Pa.z, i);
              const float lx = __shfl_sync(0xffffffffu, Qa.x, i), ly = __shfl_sync(0xffffffffu, Qa.y, i),
                          lz = __shfl_sync(0xffffffffu, Qa.z, i);
              const float e2i = __shfl_sync(0xffffffffu, (float)eps2, i);
              const int32_t ai = __shfl_sync(0xffffffffu, a, i);
              float fx = 0.f, fy = 0.f, fz = 0.f;
              bool ok = false;
              if (lane < c && bm != ai) {
                const float dx = (ax - pb.x) + (lx - qb.x), dy = (ay - pb.y) + (ly - qb.y),
                            dz = (az - pb.z) + (lz - qb.z);
                const float q = norm2(dx, dy, dz) + e2i;
                if (q > 0.f) {
                  const float gq = gmk * inv_q32(q);
                  fx = gq * dx;
                  fy = gq * dy;
                  fz = gq * dz;
                  ok = true;
                }
              }
              for (int o = 16; o > 0; o >>= 1) {
                fx += __shfl_xor_sync(0xffffffffu, fx, o);
                fy += __shfl_xor_sync(0xffffffffu, fy, o);
                fz += __shfl_xor_sync(0xffffffffu, fz, o);
              }
              const unsigned okm = __ballot_sync(0xffffffffu, ok);
              if (lane == i) {
                acc.add((R)fx, (R)fy, dim == 3 ? (R)fz : R(0));
                if constexpr (COUNT) nterm += __popc(okm);
              }
            }
          } else if (direct) {
            for (int k = 0; k < c; ++k) {
              if (base + k == slot) continue;  // the particle itself
              R d[3], gm;  // gm = -G m_b
              const float4 ph = sh_hi[w][k], pl = sh_lo[w][k];
              d[0] = (Pa.x - ph.x) + (Qa.x - pl.x);
              d[1] = (Pa.y - ph.y) + (Qa.y - pl.y);
              d[2] = (Pa.z - ph.z) + (Qa.z - pl.z);
              gm = ph.w;
              const R r2 = norm2(d[0], d[1], d[2]);
              const R q = r2 + eps2;
              if (!(q > R(0))) continue;
              const R gq = gm * inv_q32(q);
              acc.add_scaled(gq, d);
              if constexpr (COUNT) ++nterm;
            }
          }
          __syncwarp();
        }
      }
    }
    if (iter > nnodes) raise_err(A.err, ERR_TIMEOUT);
    if (COUNT && A.ctr) {
      warp_count(A.ctr + CTR_GRAV_NODES, nacc);
      warp_count(A.ctr + CTR_GRAV_TERMS, nterm);
      if (lane == 0) atomicAdd(A.ctr + CTR_GRAV_VISITS, (unsigned long long)iter);
    }
    if (act) {
      double gx, gy, gz;
      acc.value(gx, gy, gz);
      const double osc = A.U->acc;
      A.out[0][a] = gx * osc;
      A.out[1][a] = gy * osc;
      if (DIM == 3) A.out[2][a] = gz * osc;
    }
  }
}

// ---------------------------------------------------------------------------
// FP64 walk.  Bound by the FP64 unit (a warp instruction every 16 cycles per
// SM), so the walk itself spends none of it and the terms run on full warps:
//  - acceptance as in the mixed walk, in FP32 with the FP64 expression inside
//    a band of 1e-4 (far above the FP32 error): the same accepted set;
//  - a lane appends what it accepts (nodes) and what it sums directly (leaf
//    members) to its own list in shared memory; when a list may overflow the
//    warp evaluates all lists in lockstep.  Evaluated where they are met, a
//    term would occupy the unit for the 18 of 32 lanes that accept the node;
//  - a term takes 17 FP64 instructions, with rsqrt64 in place of a square root
//    and a division, and G applied to the sums.
// A lane's terms are summed in the order of its own walk, whatever the warp.
// 50k cloud, the whole call: 9.05 -> 2.57 ms (before: acceptance and terms in FP64
// at the node, about 45 instructions each).
// ---------------------------------------------------------------------------
constexpr int kList64 = 64;  // entries per lane: a leaf's 32 members fit while 32 wait

template <int DIM>
__global__ void __launch_bounds__(32, kGrav64Blocks) k_gravity64(GravArgs A) {
  __shared__ int32_t list[kList64][32];  // node id, or ~particle
  const Tree &T = A.T;
  const int lane = threadIdx.x & 31;
  // lane `sub` of the 2^share lanes of a particle takes its terms sub, sub + 2^share, ...
  const int share = A.share, sub = lane & ((1 << share) - 1), every = (1 << share) - 1;
  const bool chunks = T.ninst <= 1;
  const int per = 32 >> share;  // particles of a chunk
  const int ngroups = chunks ? (int)((T.n + per - 1) / per) : *T.ngroups;
  const int L = T.leaf_size, B = T.max_depth;
  const int nnodes = T.iter_cap > 0 ? min(*T.nnodes, T.iter_cap) : *T.nnodes;
  const int64_t cap = T.cap_nodes;
  const double th = A.theta;
  const float th2f = (float)(th * th);
  const bool test_inside = A.test_inside != 0;
  for (int g = blockIdx.x; g < ngroups; g += gridDim.x) {
    const int32_t s0 = chunks ? g * per : T.grp_start[g];
    const int32_t s1 = chunks ? (int32_t)(((int64_t)s0 + per < T.n) ? (int64_t)s0 + per : T.n) : T.grp_end[g];
    const int inst = chunks ? 0 : T.grp_inst[g];
    const int32_t slot = s0 + (lane >> share);
    const bool act = slot < s1;
    const int32_t a = act ? (T.perm_identity ? slot : T.perm[slot]) : 0;
    double xa[3] = {0.0, 0.0, 0.0}, acc[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int ax = 0; ax < DIM; ++ax) xa[ax] = A.x[ax][a];
    const unsigned long long ka =
        !act || !test_inside
            ? 0ULL
            : (A.reuse ? morton_key(xa, DIM, B, inst, T.inst_lo, T.inst_s0[inst], T.inst_rs0[inst]) : T.skey[slot]);
    const float4 Pa = A.pk.px(a), Qa = A.pk.pxl(a);
    const double e = A.eps * A.h[a], eps2 = e * e;
    const float s0f = to_f32_scaled(T.inst_s0[inst], pow2_exp(A.U->invL), A.U->invL);
    const int32_t root = T.inst_root[inst];
    const int32_t stop = root >= 0 ? T.skip[root] : root;
    int32_t skip_until = -1;
    int len = 0, iter = 0, met = 0;  // met: terms of this particle, on all its lanes
    unsigned nacc = 0, nterm = 0;
    auto evaluate = [&]() {
      double p[DIM], m = 0.0;
      int32_t ent = 0;
      auto fetch = [&](int k) {
        ent = list[k][lane];
        const bool part = ent < 0;
        const int64_t i = part ? ~ent : ent;
#pragma unroll
        for (int ax = 0; ax < DIM; ++ax) p[ax] = part ? A.x[ax][i] : T.com[ax * cap + i];
        m = part ? A.m[i] : T.mass[i];
      };
      if (len > 0) fetch(0);
      for (int k = 0; k < len; ++k) {
        double d[DIM], q = eps2;
        const double mk = m;
#pragma unroll
        for (int ax = 0; ax < DIM; ++ax) {
          d[ax] = xa[ax] - p[ax];
          q = fma(d[ax], d[ax], q);
        }
        nterm += (unsigned)(ent < 0 && (int64_t)dbits(q) > 0);
        if (k + 1 < len) fetch(k + 1);
        const double y = rsqrt64(q);  // 0 where q = 0
        const double f = mk * y * (y * y);
#pragma unroll
        for (int ax = 0; ax < DIM; ++ax) acc[ax] = fma(f, d[ax], acc[ax]);
      }
      len = 0;
      __syncwarp();
    };
    for (int32_t nd = root; nd < stop && iter <= nnodes; ++iter) {
      const int4 rec = __ldg(&T.nrec[nd]);  // (first, end, skip, level)
      const float4 ch = __ldg(&T.fcom_hi[nd]), cl = __ldg(&T.fcom_lo[nd]);
      const bool leaf = rec.y - rec.x <= L || rec.w == B;
      bool open = false, direct = false;
      if (act && nd >= skip_until) {
        bool accept = false;
        if (!(test_inside && (ka >> (DIM * (B - rec.w))) == T.cell[nd])) {
          const float dx = (Pa.x - ch.x) + (Qa.x - cl.x), dy = (Pa.y - ch.y) + (Qa.y - cl.y),
                      dz = (Pa.z - ch.z) + (Qa.z - cl.z);
          const float sf = __int_as_float(__float_as_int(s0f) - (rec.w << 23));
          const float lhs = sf * sf, rhs = th2f * (dx * dx + dy * dy + dz * dz);
          if (lhs < rhs * (1.0f - kMacBand) && rhs < 1e37f && lhs > 1e-30f) accept = true;
          else if (lhs > rhs * (1.0f + kMacBand) && lhs < 1e37f && lhs > 1e-30f) accept = false;
          else  // rare: the FP64 decision
            accept = ldexp(T.inst_s0[inst], -rec.w) <
                     th * sqrt(r2_fp64<DIM>(xa, T.com[nd], T.com[cap + nd], DIM == 3 ? T.com[2 * cap + nd] : 0.0));
        }
        if (accept) {
          if ((met++ & every) == sub) {
            list[len++][lane] = nd;
            ++nacc;
          }
          skip_until = rec.z;
        } else if (leaf) {
          direct = true;
          skip_until = rec.z;
        } else {
          open = true;
        }
      }
      const bool any_open = __any_sync(0xffffffffu, open);
      if (__any_sync(0xffffffffu, direct)) {
        for (int32_t base = rec.x; base < rec.y; base += kMaxLeaf) {
          const int c = min(rec.y - base, kMaxLeaf);
          if (__any_sync(0xffffffffu, len > kList64 - kMaxLeaf)) evaluate();
          const int32_t bm = lane < c ? (T.perm_identity ? base + lane : T.perm[base + lane]) : -1;
          for (int k = 0; k < c; ++k) {
            const int32_t b = __shfl_sync(0xffffffffu, bm, k);
            if (direct && b != a && (met++ & every) == sub) list[len++][lane] = ~b;
          }
        }
      }
      if (__any_sync(0xffffffffu, len == kList64)) evaluate();
      nd = any_open ? nd + 1 : rec.z;
    }
    evaluate();
    if (iter > nnodes) raise_err(A.err, ERR_TIMEOUT);
    if (A.ctr) {
      warp_count(A.ctr + CTR_GRAV_NODES, nacc);
      warp_count(A.ctr + CTR_GRAV_TERMS, nterm);
      if (lane == 0) atomicAdd(A.ctr + CTR_GRAV_VISITS, (unsigned long long)iter);
    }
    for (int o = 1; o <= every; o <<= 1)
#pragma unroll
      for (int ax = 0; ax < DIM; ++ax) acc[ax] += __shfl_xor_sync(0xffffffffu, acc[ax], o);
    if (act && sub == 0) {
#pragma unroll
      for (int ax = 0; ax < DIM; ++ax) A.out[ax][a] = -A.G * acc[ax];
    }
  }
}

template <int DIM>
static void gravity_mixed(const GravArgs &A, bool packed, int blocks, cudaStream_t st) {
  const int threads = kGrWarps * 32;
  if (!packed) k_gravity<DIM, false, true, true><<<blocks, threads, 0, st>>>(A);
  else if (A.ctr) k_gravity<DIM, true, true, true><<<blocks, threads, 0, st>>>(A);
  else if (A.test_inside) k_gravity<DIM, true, true, false><<<blocks, threads, 0, st>>>(A);
  else k_gravity<DIM, true, false, false><<<blocks, threads, 0, st>>>(A);
}

void gravity_walk(sph_ctx *c, const sph_state *s, const sph_params &p, double *ax, double *ay, double *az,
                  cudaStream_t st, bool reuse) {
  if (s->n == 0) return;
  GravArgs A;
  memset(&A, 0, sizeof(A));
  A.T = c->tree;
  A.pk = c->pk;
  for (int k = 0; k < 3; ++k) A.x[k] = s->x[k];
  A.m = s->m;
  A.h = s->h;
  A.dim = s->dim;
  A.G = p.G;
  A.theta = p.theta;
  A.eps = p.eps_grav;
  A.out[0] = ax;
  A.out[1] = ay;
  A.out[2] = az;
  A.U = c->units;
  A.err = c->d_err;
  A.reuse = reuse ? 1 : 0;
  A.test_inside = (double)s->dim * p.theta * p.theta >= 0.99;
  A.ctr = counters(c);
  // One instance: a block per chunk, so that the hardware hands chunks out as
  // warps finish (a persistent grid gave each block every 4864th chunk: at 400k
  // two or three of them, and a last wave a sixth full; 2M cloud step 39.7 ->
  // 36.9 ms, 400k pair window 21.3 -> 19.9 ms).  Several: the number of groups
  // is only known on the device, and the resident blocks loop over them.
  const int blocks = c->tree.ninst <= 1 ? nblk(s->n, 32 * kGrWarps) : c->num_sms * SPH_GRAV_MIN_BLOCKS;
  const bool mixed = p.precision == SPH_MIXED;
  // FP64, one instance: two lanes share a particle (a warp then walks for 16
  // particles, whose lists fill evenly), four or eight where those still fit
  // one wave of resident warps.  One, two, four, eight lanes: 10k cloud -,
  // 1.58, 1.36, 1.38 ms; 50k 3.9, 3.14, 3.42, 4.28; 200k 14.4, 11.6, 10.8,
  // 14.1; 1M 64, 55.6, 58.5, 85.4 ms.
  A.share = !mixed && c->tree.ninst <= 1 ? 1 : 0;
  while (A.share > 0 && A.share < 3 && (s->n << (A.share + 1)) <= (int64_t)32 * 32 * c->num_sms) ++A.share;
  const bool packed = mixed && c->tree.packed_walk;
  const int blocks64 = c->tree.ninst <= 1 ? nblk(s->n << A.share, 32) : c->num_sms * kGrav64Blocks;
  if (s->dim == 3) {
    if (mixed) gravity_mixed<3>(A, packed, blocks, st);
    else k_gravity64<3><<<blocks64, 32, 0, st>>>(A);
  } else {
    if (mixed) gravity_mixed<2>(A, packed, blocks, st);
    else k_gravity64<2><<<blocks64, 32, 0, st>>>(A);
  }
  ++sph::g_launches;
}

}  // namespace sph
