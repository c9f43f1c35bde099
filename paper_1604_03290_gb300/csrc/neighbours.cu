// Interaction partners (Sect. 3.5.2), GB300 form.
//
// The paper walks the tree once per particle from the root.  Here a warp
// walks it once for a group of up to 32 particles of sibling cells, 32 nodes
// at a time, a lane each.  A node is entered when its particle box comes
// within (h_group + h_node,max)/2 of the group's box, which can only keep
// more candidates than the paper's test; the set itself is decided per lane
// by the exact predicate.
//
// Predicate: b is a partner of a iff ((dx^2 + dy^2) + dz^2) < h_ab^2 with
// h_ab = (h_a + h_b)/2, all in FP64 without fused multiply-add.  On GB300
// FP64 runs at 1/62 of the FP32 rate, so each candidate is first classified
// in FP32 from positions relative to the group (formed from hi/lo split
// coordinates); only candidates whose squared distance lies within a
// relative band of 6e-5 around h_ab^2 - far wider than the FP32 error of
// about 2e-6 - are decided by the FP64 expression.  The result is therefore
// bit-identical to the FP64 definition.
#include <algorithm>
#include <climits>

#include "fpbits.cuh"
#include "sph_internal.cuh"

namespace sph {

// Warps (particle groups) per block; the grid keeps the warp count of 4-warp
// blocks.  1, 2 and 4 measured within 3 % of each other on GB300.
#ifndef SPH_WALK_WARPS
#define SPH_WALK_WARPS 4
#endif
constexpr int kNbWarps = SPH_WALK_WARPS;
// resident blocks per SM the walk is compiled for: at 8 (64 registers) it
// spills, 5 and 6 are equally fast at 1M and 5 is faster at small n (a 14k RK3
// call 2.84 against 2.89 ms)
#ifndef SPH_WALK_MIN_BLOCKS
#define SPH_WALK_MIN_BLOCKS 5
#endif
#define SPH_WALK_BOUNDS __launch_bounds__(kNbWarps * 32, SPH_WALK_MIN_BLOCKS)
constexpr float kBand = 6e-5f;

__device__ __forceinline__ bool exact_partner(const double *__restrict__ x, const double *__restrict__ y,
                                              const double *__restrict__ z, const double *__restrict__ h, int dim,
                                              int64_t a, int64_t b) {
  double dx = __dsub_rn(x[a], x[b]);
  double dy = __dsub_rn(y[a], y[b]);
  double r2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
  if (dim == 3) {
    double dz = __dsub_rn(z[a], z[b]);
    r2 = __dadd_rn(r2, __dmul_rn(dz, dz));
  }
  double hab = __dmul_rn(0.5, __dadd_rn(h[a], h[b]));
  return r2 < __dmul_rn(hab, hab);
}

// The same predicate with the particle's own support radius, for the
// variable smoothing length iteration: ((dx^2 + dy^2) + dz^2) < h_a^2.
__device__ __forceinline__ bool exact_within_own_h(const double *__restrict__ x, const double *__restrict__ y,
                                                   const double *__restrict__ z, const double *__restrict__ h,
                                                   int dim, int64_t a, int64_t b) {
  double dx = __dsub_rn(x[a], x[b]);
  double dy = __dsub_rn(y[a], y[b]);
  double r2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
  if (dim == 3) {
    double dz = __dsub_rn(z[a], z[b]);
    r2 = __dadd_rn(r2, __dmul_rn(dz, dz));
  }
  return r2 < __dmul_rn(h[a], h[a]);
}

// Shells (SHELL = true): the walk also records, in ascending order, every b
// with (1 - kSkin) h_ab <= r_ab < (1 + kSkin) h_ab (FP32 tests with the band's
// margin on both sides, so possibly a few more): the partners near the
// support radius and the non-partners just beyond it, for k_partners_refine.
constexpr float kSkinF = (float)kSkin;
constexpr float kShell2 = (1.0f + kSkinF) * (1.0f + kSkinF) * (1.0f + kBand);
constexpr float kInner2 = (1.0f - kSkinF) * (1.0f - kSkinF) * (1.0f - kBand);

// ---------------------------------------------------------------------------
// The walk.  A warp takes one group (<= 32 particles of sibling cells) and
//  1. finds the nodes where the walk stops (flagged in their box word) whose
//     box comes within reach of the group's: a stack of nodes in shared
//     memory, up to 32 popped and tested at once, one per lane, their children
//     pushed together.  The ranges found are then sorted by their first slot,
//     so that partners come out ascending whatever the order of the tests;
//  2. streams the ranges' particles as one sequence, 32 at a time across range
//     ends, and keeps those within reach of the group's box;
//  3. tests the kept candidates, 33 to 64 at a time, against every lane's own
//     particle.
// Visiting the nodes one after the other, as a single particle would, cost
// 146 dependent visits per group on the 1M impact, each a round trip to the
// L1 or L2, and a separate round of loads and a separate test loop for every
// range: 1.11 ms there (now 0.80), 0.40 ms with shells at 263k (now 0.26, half
// of the difference by the tickets), 84 us for the 600 groups of a 14k body
// (now 70).  Issue-bound at 1M (0.62G warp instructions).  Tried and left out:
// two or four lanes per particle at small n (1 % of an RK3 call).
// More ranges or nodes than the shared buffers hold: the ranges of that group
// come from a one-by-one walk in slot order instead, consumed as the buffer
// fills.
// ---------------------------------------------------------------------------
constexpr int kWalkStack = 384;   // nodes
constexpr int kWalkRanges = 128;  // ranges of one group
constexpr int kWalkCand = 64;     // kept candidates (tested when more than 32 wait)
struct WalkScratch {
  union {
    int32_t stack[kWalkStack];
    struct {
      float4 c[kWalkCand];  // position relative to the group's reference, half its support radius
      int32_t b[kWalkCand];
    } cand;
  };
  int32_t first[kWalkRanges], count[kWalkRanges];    // as found
  int32_t sfirst[kWalkRanges], soff[kWalkRanges];    // sorted: first slot, and number of particles before
};

// Ranges of a group, sorted by first slot, with the running particle count;
// returns the total.
__device__ __forceinline__ int32_t sort_ranges(WalkScratch &W, int nr, int lane) {
  int32_t f[kWalkRanges / 32], r[kWalkRanges / 32];
#pragma unroll
  for (int j = 0; j < kWalkRanges / 32; ++j) {
    f[j] = 32 * j + lane < nr ? W.first[32 * j + lane] : INT_MAX;
    r[j] = 0;
  }
  for (int t = 0; t < nr; ++t) {
    const int32_t k = W.first[t];
#pragma unroll
    for (int j = 0; j < kWalkRanges / 32; ++j)
      if (32 * j < nr) r[j] += k < f[j];
  }
#pragma unroll
  for (int j = 0; j < kWalkRanges / 32; ++j)
    if (32 * j + lane < nr) {
      W.sfirst[r[j]] = f[j];
      W.soff[r[j]] = W.count[32 * j + lane];
    }
  __syncwarp();
  int32_t total = 0;
  for (int j = 0; j < nr; j += 32) {
    const int32_t v = j + lane < nr ? W.soff[j + lane] : 0;
    int32_t incl = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    if (j + lane < nr) W.soff[j + lane] = total + incl - v;
    total += __shfl_sync(0xffffffffu, incl, 31);
  }
  __syncwarp();
  return total;
}

// Groups a refine queues for walking again: two queues (phases), a bit per
// group in each so that a group is queued once.  Words: the two counts, then
// the bits; the queues lie in Tree::arrived, free after a build.
struct Redo {
  int32_t *w;
  int32_t *q;
  int64_t words, cap;  // bit words and entries per queue
  __device__ __forceinline__ int32_t *queue(int phase) const { return q + (phase - 1) * cap; }
  __device__ __forceinline__ int count(int phase) const { return w[phase - 1]; }
  __device__ __forceinline__ int32_t *bits(int phase, int g) const { return w + 4 + (phase - 1) * words + (g >> 5); }
  __device__ __forceinline__ bool queued(int phase, int g) const {
    return (*(const volatile int32_t *)bits(phase, g) >> (g & 31)) & 1;
  }
  // queue group g, unless it is `own` (or for phase 2 already in phase 1)
  __device__ __forceinline__ void add(int phase, int g, int own) const {
    if (g == own || queued(phase, g) || (phase == 2 && queued(1, g))) return;
    const int32_t bit = (int32_t)(1u << (g & 31));
    if (atomicOr(bits(phase, g), bit) & bit) return;
    queue(phase)[atomicAdd(&w[phase - 1], 1)] = g;
  }
};
int64_t redo_words(int64_t cap_groups) { return 4 + 2 * ((cap_groups + 31) / 32); }

// A particle whose own displacement bound since the walk allows the refine
// (see k_partners_refine): 2 sqrt(D) disp <= kSkin h, in code units; the FP32
// rounding of h (2^-24) and of the products is in the factor.
__device__ __forceinline__ bool slow_particle(float disp, float h, int dim) {
  const float f = dim == 3 ? 2.0f * 1.7320508f * (1.0f + 1e-5f) : 2.0f * 1.4142136f * (1.0f + 1e-5f);
  return __fmul_ru(f, disp) <= __fmul_rd(kSkinF, h);
}

// OWN_H = false: interaction partners (h_ab), lists and counts.  OWN_H = true:
// only the number of particles within each particle's own h (the current h of
// the state, not the packed one), plus the count of particles whose number
// lies farther than tol from n_des (*unconverged); the walk is skipped once
// *done is set.
// Warps draw their groups from a ticket counter (tick[0]): a fixed stride left
// half the warps a second group and the others none at 263k particles.  The
// last warp to find no group left (tick[1] counts them) sets both back to 0.
// SELECT (after a refine): only the groups queued for walking again, all their
// particles.  Phase 1 takes the first queue (groups of particles that could
// not refine their lists) and, of particles that moved too far, queues the
// groups of the partners they had and of those they have now; phase 2 takes
// these where phase 1 has not walked them.  With more than half of the groups
// in the first queue, or few enough that each warp takes one (the walk then
// lasts as long as its slowest group), phase 1 walks them all and phase 2
// none.  SHELL records each particle's group.
template <bool OWN_H, bool SHELL, bool SELECT>
__global__ void SPH_WALK_BOUNDS k_partners(Tree T, PackedF32 pk, const double *__restrict__ x,
                                           const double *__restrict__ y, const double *__restrict__ z,
                                           const double *__restrict__ h, int dim, int kmax,
                                           int32_t *__restrict__ nb_idx, int32_t *__restrict__ nb_cnt, int64_t ld,
                                           int32_t *err, const unsigned long long *__restrict__ grow,
                                           const Units *__restrict__ U, const int32_t *__restrict__ done,
                                           int32_t *__restrict__ unconverged, double n_des, int tol,
                                           int32_t *__restrict__ sh_idx, int32_t *__restrict__ sh_cnt,
                                           int32_t *__restrict__ sh_in, int32_t *tick, int32_t *grp_of, Redo R,
                                           int phase, const float *disp, const int32_t *old_idx,
                                           const int32_t *old_cnt, unsigned long long *ctr) {
  static_assert(!(OWN_H && SHELL) && !(SELECT && (OWN_H || SHELL)), "shells are partner candidates");
  if constexpr (OWN_H) {
    if (*done) return;
  }
  bool every = false;  // SELECT: every group after all
  if constexpr (SELECT) {
    every = 2 * R.count(1) > *T.ngroups || *T.ngroups <= (int)(gridDim.x * kNbWarps);
    if (R.count(phase) == 0 || (phase == 2 && every)) return;
  }
  // the shell widens every test by the factor (1 + kSkin) of its radius
  const float wide = SHELL ? 1.0f + kSkinF : 1.0f;
  __shared__ WalkScratch scratch[kNbWarps];
  WalkScratch &W = scratch[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int ngroups = SELECT && !every ? R.count(phase) : *T.ngroups;
  // The walk stops at nodes flagged in their box word (at most
  // max(leaf_size, walk_leaf) particles, or depth B; set by the tree build)
  // and culls their whole particle range: any stopping rule gives the same set.
  const int nnodes = T.iter_cap > 0 ? min(*T.nnodes, T.iter_cap) : *T.nnodes;
  // Node boxes are those of the tree the walk runs on; when the particles have
  // moved since it was built (by at most `grow` per axis), widening the
  // group's box by that much keeps every node that may hold a partner.
  float gw = 0.f;
  if (grow) gw = to_f32_dir_scaled(bitsd(*grow), pow2_exp(U->invL), true, U->invL);
  for (;;) {
    int g = 0;
    if (lane == 0) g = atomicAdd(&tick[0], 1);
    g = __shfl_sync(0xffffffffu, g, 0);
    if (g >= ngroups) break;
    if constexpr (SELECT)
      if (!every) {
        g = R.queue(phase)[g];
        if (phase == 2 && R.queued(1, g)) continue;
      }
    const int32_t s0 = T.grp_start[g], s1 = T.grp_end[g], inst = T.grp_inst[g];
    const int32_t slot = s0 + lane;
    const bool act = slot < s1;
    const int32_t a = act ? (T.perm_identity ? slot : T.perm[slot]) : -1;
    if constexpr (SHELL)
      if (act) grp_of[a] = g;
    // this lane's particle moved too far: its partners' groups are walked too
    const bool far = SELECT && act && !every && phase == 1 && !slow_particle(disp[a], pk.px(a).w, dim);
    if (far) {
      int last = g;  // neighbouring entries mostly share a group
      const int k1 = old_cnt[a];
      for (int k = 0; k < k1; ++k) {
        const int e = grp_of[old_idx[(int64_t)k * ld + a]];
        if (e != last) R.add(2, e, g);
        last = e;
      }
    }
    float4 P = act ? pk.px(a) : make_float4(0.f, 0.f, 0.f, 0.f);
    float4 Q = act ? pk.pxl(a) : make_float4(0.f, 0.f, 0.f, 0.f);
    // reference point: lane 0's position
    const float cx = __shfl_sync(0xffffffffu, P.x, 0), cy = __shfl_sync(0xffffffffu, P.y, 0),
                cz = __shfl_sync(0xffffffffu, P.z, 0);
    const float lx = __shfl_sync(0xffffffffu, Q.x, 0), ly = __shfl_sync(0xffffffffu, Q.y, 0),
                lz = __shfl_sync(0xffffffffu, Q.z, 0);
    const float rax = (P.x - cx) + (Q.x - lx), ray = (P.y - cy) + (Q.y - ly), raz = (P.z - cz) + (Q.z - lz);
    const float hha = 0.5f * P.w;
    // own support radius in code units (OWN_H): from the state's current h
    float hown = 0.f;
    if constexpr (OWN_H) hown = act ? to_f32_scaled(h[a], pow2_exp(U->invL), U->invL) : 0.f;
    // group box (hi coordinates, for the node test) and largest h
    float gl[3] = {act ? P.x : 3e38f, act ? P.y : 3e38f, act ? P.z : 3e38f};
    float gh[3] = {act ? P.x : -3e38f, act ? P.y : -3e38f, act ? P.z : -3e38f};
    float hg = act ? (OWN_H ? hown : P.w) : 0.f;
    // the same box relative to the reference point, for culling candidates
    float rl[3] = {act ? rax : 3e38f, act ? ray : 3e38f, act ? raz : 3e38f};
    float rh[3] = {act ? rax : -3e38f, act ? ray : -3e38f, act ? raz : -3e38f};
    for (int o = 16; o > 0; o >>= 1) {
      for (int ax = 0; ax < 3; ++ax) {
        gl[ax] = fminf(gl[ax], __shfl_xor_sync(0xffffffffu, gl[ax], o));
        gh[ax] = fmaxf(gh[ax], __shfl_xor_sync(0xffffffffu, gh[ax], o));
        rl[ax] = fminf(rl[ax], __shfl_xor_sync(0xffffffffu, rl[ax], o));
        rh[ax] = fmaxf(rh[ax], __shfl_xor_sync(0xffffffffu, rh[ax], o));
      }
      hg = fmaxf(hg, __shfl_xor_sync(0xffffffffu, hg, o));
    }
    float mag = fmaxf(fmaxf(fabsf(gh[0]), fabsf(gh[1])), fabsf(gh[2]));
    float slack = 1e-6f * mag + gw * (1.0f + 1e-6f);
    for (int ax = 0; ax < 3; ++ax) {
      gl[ax] -= slack;
      gh[ax] += slack;
    }
    // relative coordinates carry an error of a few 1e-7 of the group's extent + h
    const float rslack = 1e-5f * (fmaxf(fmaxf(rh[0] - rl[0], rh[1] - rl[1]), rh[2] - rl[2]) + hg);
    const int32_t root = T.inst_root[inst];
    // a square of the support that FP32 cannot hold (h infinite, or not a number)
    // tells no candidate from the padding of the test: no shell, always walked
    int cnt = 0, scnt = SHELL && !(hha * hha * kShell2 < INFINITY) ? kMaxShell + 1 : 0;
    uint32_t sin = 0;  // shell entries that are partners (bit per entry)
    unsigned ntest = 0;  // candidates this lane tested (counters)
    int32_t *out = nb_idx + a, *sout = SHELL ? sh_idx + a : nullptr;  // a = -1 writes nothing

    // a node's box words: is it within reach, and where does the walk go on
    auto reached = [&](const float4 &bl, const float4 &bh) {
      const float hw = fabsf(bl.w);
      float gx = fmaxf(0.f, fmaxf(bl.x - gh[0], gl[0] - bh.x));
      float gy = fmaxf(0.f, fmaxf(bl.y - gh[1], gl[1] - bh.y));
      float gz = fmaxf(0.f, fmaxf(bl.z - gh[2], gl[2] - bh.z));
      float d2 = gx * gx + gy * gy + gz * gz;
      float thr = (OWN_H ? hg : 0.5f * (hg + hw)) * (1.0f + 1e-5f) * wide;
      return d2 <= thr * thr;
    };
    // 3. the kept candidates against every lane's particle, four at a time
    // (one round of shared loads, four independent distances); the buffer is
    // padded with candidates out of everyone's reach and of index -2, which
    // never count: a lane with a position that is not a number or an infinite
    // h cannot tell them from its partners by distance
    auto test = [&](int nc) {
      const int np = (nc + 3) & ~3;
      if (lane < np - nc) {
        W.cand.c[nc + lane] = make_float4(3e38f, 3e38f, 3e38f, 0.f);
        W.cand.b[nc + lane] = -2;
      }
      __syncwarp();
      if (act) {
        ntest += nc;
        for (int k = 0; k < np; k += 4) {
          const int4 b4 = *reinterpret_cast<const int4 *>(&W.cand.b[k]);
          const int32_t bs[4] = {b4.x, b4.y, b4.z, b4.w};
          float r2[4], h2[4];
          bool in[4];
          unsigned unsure = 0;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 cb = W.cand.c[k + u];
            float dx = rax - cb.x, dy = ray - cb.y, dz = raz - cb.z;
            r2[u] = dx * dx + dy * dy + dz * dz;
            float hab = OWN_H ? hown : hha + cb.w;
            h2[u] = hab * hab;
            in[u] = r2[u] < h2[u] * (1.0f - kBand);
            if (!in[u] && !(r2[u] > h2[u] * (1.0f + kBand))) unsure |= 1u << u;
          }
          if (unsure) {  // rare: the FP64 predicate
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (((unsure >> u) & 1u) && bs[u] >= 0)
                in[u] = OWN_H ? exact_within_own_h(x, y, z, h, dim, a, bs[u]) : exact_partner(x, y, z, h, dim, a, bs[u]);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const bool other = bs[u] != a;
            if (in[u] && other) {
              if constexpr (!OWN_H) {
                if (cnt < kmax) *out = bs[u];
                out += ld;
              }
              if constexpr (SELECT)
                if (far) R.add(2, grp_of[bs[u]], g);
              ++cnt;
            }
            if constexpr (SHELL) {
              // near the support radius on either side
              if (other && r2[u] >= h2[u] * kInner2 && r2[u] <= h2[u] * kShell2) {
                if (scnt < kMaxShell) {
                  *sout = bs[u];
                  sin |= (uint32_t)in[u] << scnt;
                }
                sout += ld;
                ++scnt;
              }
            }
          }
        }
      }
      __syncwarp();
    };
    // 2. the particles of nr ranges (sorted), culled against the group's box
    auto consume = [&](int nr, int32_t total) {
      int i = 0, kept = 0;  // i: this lane's range
      int32_t b = -1;
      float4 Pb, Qb;
      auto load = [&](int32_t flat) {
        b = -1;
        if (flat < total) {
          while (i + 1 < nr && W.soff[i + 1] <= flat) ++i;
          const int32_t sl = W.sfirst[i] + (flat - W.soff[i]);
          b = T.perm_identity ? sl : __ldg(&T.perm[sl]);
          Pb = __ldg(&pk.px(b));
          Qb = __ldg(&pk.pxl(b));
        }
      };
      load(lane);
      for (int32_t base = 0; base < total; base += 32) {
        bool keep = false;
        const int32_t bk = b;
        float4 cand = make_float4(0.f, 0.f, 0.f, 0.f);
        if (bk >= 0) {
          cand = make_float4((Pb.x - cx) + (Qb.x - lx), (Pb.y - cy) + (Qb.y - ly), (Pb.z - cz) + (Qb.z - lz),
                             0.5f * Pb.w);  // half support radius: h_ab = h_a / 2 + h_b / 2
          float qx = fmaxf(0.f, fmaxf(rl[0] - cand.x, cand.x - rh[0]));
          float qy = fmaxf(0.f, fmaxf(rl[1] - cand.y, cand.y - rh[1]));
          float qz = fmaxf(0.f, fmaxf(rl[2] - cand.z, cand.z - rh[2]));
          float reach = (OWN_H ? hg : 0.5f * hg + cand.w) * (1.0f + 1e-5f) * wide + rslack;
          keep = qx * qx + qy * qy + qz * qz <= reach * reach;
        }
        load(base + 32 + lane);  // the next 32, in flight during the tests
        const unsigned km = __ballot_sync(0xffffffffu, keep);
        if (keep) {
          const int pos = kept + __popc(km & lt_mask);
          W.cand.c[pos] = cand;
          W.cand.b[pos] = bk;
        }
        kept += __popc(km);
        if (kept > kWalkCand - 32) {
          test(kept);
          kept = 0;
        }
      }
      if (kept) test(kept);
    };

    // 1. the ranges within reach
    int nr = 0, visited = 0;
    bool fits = true;
    if (root >= 0) {
      int sp = 1;
      if (lane == 0) W.stack[0] = root;
      __syncwarp();
      while (sp > 0 && visited <= nnodes) {
        const int m = min(sp, 32);
        const int32_t nd = lane < m ? W.stack[sp - m + lane] : -1;
        sp -= m;
        visited += m;
        __syncwarp();
        bool hit = false;
        int nc = 0;
        int4 rec = make_int4(0, 0, 0, 0), c0 = make_int4(-1, -1, -1, -1), c1 = c0;
        if (nd >= 0) {
          const float4 bl = __ldg(&T.fbox_lo[nd]), bh = __ldg(&T.fbox_hi[nd]);
          if (reached(bl, bh)) {
            hit = (__float_as_uint(bl.w) >> 31) != 0u;  // the walk stops here
            if (hit) {
              rec = __ldg(&T.nrec[nd]);
            } else {
              const int4 *ch = reinterpret_cast<const int4 *>(T.child) + 2 * (int64_t)nd;
              c0 = __ldg(ch);
              if (dim == 3) c1 = __ldg(ch + 1);
              nc = (c0.x >= 0) + (c0.y >= 0) + (c0.z >= 0) + (c0.w >= 0) + (c1.x >= 0) + (c1.y >= 0) + (c1.z >= 0) +
                   (c1.w >= 0);
            }
          }
        }
        const unsigned hm = __ballot_sync(0xffffffffu, hit);
        const int pos = nr + __popc(hm & lt_mask);
        if (hit && pos < kWalkRanges) {
          W.first[pos] = rec.x;
          W.count[pos] = rec.y - rec.x;
        }
        nr += __popc(hm);
        int incl = nc;  // children pushed by the lanes up to this one
        for (int o = 1; o < 32; o <<= 1) {
          const int u = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += u;
        }
        const int push = __shfl_sync(0xffffffffu, incl, 31);
        if (nr > kWalkRanges || sp + push > kWalkStack) {
          fits = false;
          break;
        }
        if (nc > 0) {
          int at = sp + incl - nc;
          const int32_t k[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (k[j] >= 0) W.stack[at++] = k[j];
        }
        sp += push;
        __syncwarp();
      }
    }
    if (fits) {
      const int32_t total = sort_ranges(W, nr, lane);
      consume(nr, total);
    } else {
      // one by one in slot order: enter a node (nd + 1) or jump its subtree
      visited = 0;
      nr = 0;
      __syncwarp();
      const int32_t stop = T.skip[root];
      for (int32_t nd = root; nd < stop && visited <= nnodes; ++visited) {
        const float4 bl = __ldg(&T.fbox_lo[nd]), bh = __ldg(&T.fbox_hi[nd]);
        bool enter = false;
        if (reached(bl, bh)) {
          if (__float_as_uint(bl.w) >> 31) {
            const int4 rec = __ldg(&T.nrec[nd]);
            if (lane == 0) {
              W.first[nr] = rec.x;
              W.count[nr] = rec.y - rec.x;
            }
            if (++nr == kWalkRanges) {
              __syncwarp();
              const int32_t total = sort_ranges(W, nr, lane);
              consume(nr, total);
              nr = 0;
            }
          } else {
            enter = true;
          }
        }
        nd = enter ? nd + 1 : __float_as_int(bh.w);
      }
      __syncwarp();
      const int32_t total = sort_ranges(W, nr, lane);
      consume(nr, total);
    }
    if (visited > nnodes) raise_err(err, ERR_TIMEOUT);
    if (ctr) {
      warp_count(ctr + CTR_WALK_TESTS, ntest);
      warp_count(ctr + CTR_WALK_PARTNERS, act && !OWN_H ? (unsigned)cnt : 0u);
    }
    if constexpr (OWN_H) {
      if (act) {
        nb_cnt[a] = cnt;
        if (fabs((double)cnt - n_des) > (double)tol) atomicAdd(unconverged, 1);
      }
    } else if (act) {
      nb_cnt[a] = min(cnt, kmax);
      if (cnt > kmax) raise_err(err, ERR_NB_OVERFLOW);
      if constexpr (SHELL) {
        sh_cnt[a] = scnt <= kMaxShell ? scnt : -1;
        sh_in[a] = (int32_t)sin;
      }
    }
  }
  if (lane == 0 && atomicAdd(&tick[1], 1) == (int)(gridDim.x * kNbWarps) - 1) {
    tick[0] = 0;
    tick[1] = 0;
  }
}

// Partners at moved positions from the lists and shells of an earlier walk
// (the Verlet-list idea).  A particle is slow when 2 sqrt(D) times the bound
// of its own largest per-axis displacement since that walk is at most kSkin
// h_a.  The distance of two slow particles changed by at most sqrt(D) (move_a
// + move_b) <= kSkin h_ab: a partner of the walk closer than (1 - kSkin) h_ab
// is still one, a non-partner farther than (1 + kSkin) h_ab is still none, and
// only the shell between the two can change.  The old list and the shell are
// both ascending, and the shell's partners are also in the list: merged, the
// candidates are visited in ascending order, the list's members outside the
// shell are kept as they are (no gather), and each shell member is decided by
// the walk's predicate (FP32 outside the band, the FP64 definition inside it),
// so the new list equals that of a walk at the new positions bit for bit.
// The groups of fast particles (and of those whose shell overflowed) are
// walked again, and so are those of every slow one whose status with a fast
// one may differ from what its list and shell say: the fast one's old
// partners and its new ones, both queued by the walk of its group (unless that
// takes every group anyway).  A projectile's
// few fast particles so cost a walk of its surroundings; taking the largest
// displacement of all particles for each, every evaluation of a batch of
// impacts walked every group (64 impacts, 8 evaluations: 3.6 of 12.6 ms, now
// 1.6 of 10.7).
constexpr int kRefineThreads = 128;
__global__ void __launch_bounds__(kRefineThreads)
    k_partners_refine(PackedF32 pk, const double *__restrict__ x, const double *__restrict__ y,
                      const double *__restrict__ z, const double *__restrict__ h, int dim, int64_t n, int64_t ld,
                      int kmax, const int32_t *__restrict__ old_idx, const int32_t *__restrict__ old_cnt,
                      const int32_t *__restrict__ sh_idx, const int32_t *__restrict__ sh_cnt,
                      const int32_t *__restrict__ sh_in, int32_t *__restrict__ new_idx,
                      int32_t *__restrict__ new_cnt, const float *__restrict__ disp,
                      const int32_t *__restrict__ grp_of, Redo R, int32_t *err) {
  // the shell of each thread's particle, staged for the merge
  __shared__ int32_t shs[kMaxShell][kRefineThreads];
  const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= n) return;
  const int ns = sh_cnt[a];
  const bool slow = slow_particle(disp[a], pk.px(a).w, dim);
  if (ns < 0 || !slow) {
    const int g = grp_of[a];  // one lane of each group queues it
    if ((threadIdx.x & 31) == (unsigned)(__ffs(__match_any_sync(__activemask(), g)) - 1)) R.add(1, g, -1);
    return;
  }
  const int t = threadIdx.x;
  // 1. decide every shell member at the new positions (bit j of `in`)
  uint32_t in = 0;
  {
    const float4 P = pk.px(a), Q = pk.pxl(a);
    const float hha = 0.5f * P.w;
    for (int j = 0; j < ns; ++j) {
      const int32_t b = sh_idx[(int64_t)j * ld + a];
      shs[j][t] = b;
      const float4 Pb = pk.px(b), Qb = pk.pxl(b);
      const float dx = (P.x - Pb.x) + (Q.x - Qb.x), dy = (P.y - Pb.y) + (Q.y - Qb.y),
                  dz = (P.z - Pb.z) + (Q.z - Qb.z);
      const float r2 = dx * dx + dy * dy + dz * dz;
      const float hab = hha + 0.5f * Pb.w;
      const float h2 = hab * hab;
      bool ok;
      if (r2 < h2 * (1.0f - kBand)) ok = true;
      else if (r2 > h2 * (1.0f + kBand)) ok = false;
      else ok = exact_partner(x, y, z, h, dim, a, b);
      in |= (uint32_t)ok << j;
    }
  }
  // 2a. no shell member changed sides: the list is the walk's, and a count of
  // -1 tells the passes to read that list (nothing is copied)
  if (in == (uint32_t)sh_in[a]) {
    new_cnt[a] = -1;
    return;
  }
  // 2b. merge: list members outside the shell are kept, shell members that are
  // in are emitted once (in the list or inserted), the others dropped; the
  // list is read 8 entries at a time so that its loads overlap
  const int nl = old_cnt[a];
  int j = 0, cnt = 0;
  int32_t bs = ns > 0 ? shs[0][t] : INT_MAX;
  auto emit = [&](int32_t b) {
    if (cnt < kmax) new_idx[(int64_t)cnt * ld + a] = b;
    ++cnt;
  };
  for (int base = 0; base < nl; base += 8) {
    int32_t buf[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) buf[u] = base + u < nl ? old_idx[(int64_t)(base + u) * ld + a] : INT_MAX;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int32_t b = buf[u];
      if (b != INT_MAX) {
        while (bs < b) {  // shell members below b that are not in the list
          if ((in >> j) & 1u) emit(bs);
          ++j;
          bs = j < ns ? shs[j][t] : INT_MAX;
        }
        if (bs == b) {  // a list member in the shell: kept if still in
          if ((in >> j) & 1u) emit(b);
          ++j;
          bs = j < ns ? shs[j][t] : INT_MAX;
        } else {
          emit(b);
        }
      }
    }
  }
  for (; j < ns; ++j)
    if ((in >> j) & 1u) emit(shs[j][t]);
  new_cnt[a] = min(cnt, kmax);
  if (cnt > kmax) raise_err(err, ERR_NB_OVERFLOW);
}

// Blocks of a walk: the resident ones, or at small n about as many warps as
// there are groups (16 particles a warp; idle warps still draw a ticket).
static int walk_grid(const sph_ctx *c, int64_t n) {
  return std::min(c->num_sms * c->tune.walk_blocks_per_sm * (4 / kNbWarps), nblk(n, 16 * kNbWarps));
}

void find_partners(sph_ctx *c, const sph_state *s, cudaStream_t st, const unsigned long long *grow, bool shell) {
  if (s->n == 0) return;
  const bool sh = shell && c->sh_idx != nullptr;
  const auto kern = sh ? k_partners<false, true, false> : k_partners<false, false, false>;
  kern<<<walk_grid(c, s->n), kNbWarps * 32, 0, st>>>(
      c->tree, c->pk, s->x[0], s->x[1], s->x[2], s->h, s->dim, c->kmax, c->nb_idx, c->nb_cnt, c->cap_n, c->d_err, grow,
      c->units, nullptr, nullptr, 0.0, 0, c->sh_idx, c->sh_cnt, c->sh_in, c->tick, c->grp_of, Redo(), 0, nullptr,
      nullptr, nullptr, counters(c));
  ++sph::g_launches;
}

void refine_partners(sph_ctx *c, const sph_state *s, const float *disp, const unsigned long long *grow,
                     cudaStream_t st) {
  const int64_t n = s->n;
  if (n == 0) return;
  // groups hold at least one particle each, so the queues fit n entries
  const Redo R{c->redo, c->tree.arrived, (c->tree.cap_groups + 31) / 32, c->tree.cap_nodes / 2};
  cudaMemsetAsync(c->redo, 0, sizeof(int32_t) * redo_words(c->tree.cap_groups), st);
  { k_partners_refine<<<nblk(n, kRefineThreads), kRefineThreads, 0, st>>>(
        c->pk, s->x[0], s->x[1], s->x[2], s->h, s->dim, n, c->cap_n, c->kmax, c->nb_idx, c->nb_cnt, c->sh_idx,
        c->sh_cnt, c->sh_in, c->nb_alt, c->nb_cnt_alt, disp, c->grp_of, R, c->d_err); ++sph::g_launches; }
  // both return at once unless a group was queued; the resident blocks only, as they usually do
  const int blocks = std::min(walk_grid(c, n), c->num_sms * SPH_WALK_MIN_BLOCKS);
  for (int phase = 1; phase <= 2; ++phase) {
    k_partners<false, false, true><<<blocks, kNbWarps * 32, 0, st>>>(
        c->tree, c->pk, s->x[0], s->x[1], s->x[2], s->h, s->dim, c->kmax, c->nb_alt, c->nb_cnt_alt, c->cap_n, c->d_err,
        grow, c->units, nullptr, nullptr, 0.0, 0, nullptr, nullptr, nullptr, c->tick, c->grp_of, R, phase, disp,
        c->nb_idx, c->nb_cnt, counters(c));
    ++sph::g_launches;
  }
}

// ---------------------------------------------------------------------------
// Variable smoothing length (Sect. 4.2): count with the own h, then
// h <- (h / 2) (1 + (n_des / n_a)^(1/D)) for every particle when any count lies
// farther than tol from n_des (else the iteration is done)
// ---------------------------------------------------------------------------
__global__ void k_h_update(double *__restrict__ h, const int32_t *__restrict__ cnt, int64_t n, int dim,
                           double n_des, const int32_t *__restrict__ unconverged, int32_t *__restrict__ done,
                           int32_t *__restrict__ updates) {
  if (*done) return;
  const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (*unconverged == 0) {
    if (a == 0) *done = 1;
    return;
  }
  if (a == 0) atomicAdd(updates, 1);
  if (a >= n) return;
  const int32_t na = cnt[a];
  if (na == 0) {
    h[a] = 2.0 * h[a];
  } else {
    const double q = n_des / (double)na;
    const double r = dim == 3 ? cbrt(q) : (dim == 2 ? sqrt(q) : q);
    h[a] = h[a] * 0.5 * (1.0 + r);
  }
}

void adapt_h(sph_ctx *c, sph_state *s, double n_des, int tol, int max_iter, int32_t *flags, cudaStream_t st) {
  // flags: [0] done, [1] updates, [2 + i] particles off target at count i
  const int64_t n = s->n;
  cudaMemsetAsync(flags, 0, sizeof(int32_t) * (max_iter + 3), st);
  if (n == 0) return;
  const int blocks = walk_grid(c, n);
  for (int i = 0; i <= max_iter; ++i) {
    { k_partners<true, false, false><<<blocks, kNbWarps * 32, 0, st>>>(c->tree, c->pk, s->x[0], s->x[1], s->x[2], s->h,
                                                               s->dim, c->kmax, c->nb_idx, c->nb_cnt, c->cap_n,
                                                               c->d_err, nullptr, c->units, flags, flags + 2 + i,
                                                               n_des, tol, nullptr, nullptr, nullptr, c->tick, nullptr, Redo(), 0, nullptr, nullptr, nullptr, nullptr); ++sph::g_launches; }
    if (i == max_iter) break;
    { k_h_update<<<nblk(n, 256), 256, 0, st>>>(s->h, c->nb_cnt, n, s->dim, n_des, flags + 2 + i, flags,
                                             flags + 1); ++sph::g_launches; }
  }
}

// ---------------------------------------------------------------------------
// CSR export (ascending within a particle)
// ---------------------------------------------------------------------------
__global__ void k_cnt_copy(const int32_t *cnt, int32_t *out, int64_t n) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = cnt[i];
  if (i == n) out[n] = 0;
}

// One warp per particle, eight neighbouring particles per block (their column
// entries share sectors).  The lists are ascending in tree slots; in state
// indices they are where the state is in tree order, and elsewhere each entry
// goes to its rank, the number of smaller entries, counted against the list
// in shared memory (up to kCsrShort entries; longer lists are read again from
// memory).  An insertion sort into global memory, a thread per particle, took
// 0.91 ms at 263k particles in lattice order, now 0.16.  The whole call for 100k
// particles of 400 partners, in tree order and in random order: 1.56 and 24.3 ms
// with the insertion sort, 1.24 and 4.31 now (4.14 in tree order while long
// lists were ranked without a look at their order).
constexpr int kCsrShort = 128;
constexpr int kCsrWarps = 8;
__global__ void __launch_bounds__(32 * kCsrWarps) k_csr_fill(const int32_t *__restrict__ nb_idx,
                                                            const int32_t *__restrict__ nb_cnt, int64_t ld,
                                                            const int64_t *__restrict__ off, int64_t n, int32_t *idx,
                                                            int64_t cap, int32_t *err) {
  __shared__ __align__(16) int32_t lists[kCsrWarps][kCsrShort];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t a = (int64_t)blockIdx.x * kCsrWarps + w;
  if (a > n) return;
  const int64_t o = off[a];
  if (a == n) {
    if (lane == 0 && o > cap) raise_err(err, ERR_CSR_OVERFLOW);
    return;
  }
  const int k = nb_cnt[a];
  if (o + k > cap) return;
  const int32_t *col = nb_idx + a;
  if (k <= kCsrShort) {
    constexpr int M = kCsrShort / 32;
    int32_t *list = lists[w];
    int32_t v[M], r[M];
#pragma unroll
    for (int j = 0; j < M; ++j) {
      v[j] = 32 * j + lane < k ? col[(int64_t)(32 * j + lane) * ld] : INT_MAX;
      list[32 * j + lane] = v[j];
      r[j] = 0;
    }
    __syncwarp();
    bool sorted = true;
#pragma unroll
    for (int j = 0; j < M; ++j)
      if (32 * j + lane + 1 < k) sorted &= v[j] < list[32 * j + lane + 1];
    if (__all_sync(0xffffffffu, sorted)) {
#pragma unroll
      for (int j = 0; j < M; ++j)
        if (32 * j + lane < k) idx[o + 32 * j + lane] = v[j];
      return;
    }
    for (int i = 0; i < k; i += 4) {  // entries beyond k are larger than any
      const int4 e = *reinterpret_cast<const int4 *>(list + i);
#pragma unroll
      for (int j = 0; j < M; ++j)
        if (32 * j < k) r[j] += (e.x < v[j]) + (e.y < v[j]) + (e.z < v[j]) + (e.w < v[j]);
    }
#pragma unroll
    for (int j = 0; j < M; ++j)
      if (32 * j + lane < k) idx[o + r[j]] = v[j];
    return;
  }
  bool sorted = true;  // ascending already: the counting below would be k^2 / 32 loads a lane
  for (int j = lane; sorted && j + 1 < k; j += 32) sorted = col[(int64_t)j * ld] < col[(int64_t)(j + 1) * ld];
  if (__all_sync(0xffffffffu, sorted)) {
    for (int j = lane; j < k; j += 32) idx[o + j] = col[(int64_t)j * ld];
    return;
  }
  for (int j = lane; j < k; j += 32) {
    const int32_t v = col[(int64_t)j * ld];
    int r = 0;
    for (int i = 0; i < k; ++i) r += col[(int64_t)i * ld] < v;
    idx[o + r] = v;
  }
}

void scan_counts(sph_ctx *c, const int32_t *in, int64_t *out, int64_t m, cudaStream_t st);

void partners_to_csr(sph_ctx *c, const sph_state *s, int64_t *off, int32_t *idx, int64_t cap, cudaStream_t st) {
  int64_t n = s->n;
  { k_cnt_copy<<<nblk(n + 1, 256), 256, 0, st>>>(c->nb_cnt, c->tree.ncount, n); ++sph::g_launches; }
  scan_counts(c, c->tree.ncount, off, n + 1, st);
  { k_csr_fill<<<nblk(n + 1, kCsrWarps), 32 * kCsrWarps, 0, st>>>(c->nb_idx, c->nb_cnt, c->cap_n, off, n, idx, cap,
                                               c->d_err); ++sph::g_launches; }
}

}  // namespace sph
