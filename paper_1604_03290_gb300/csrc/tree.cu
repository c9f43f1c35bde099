// Octree over Morton-sorted particles (Sect. 3.5.1), GB300 form.
//
// Instead of the paper's lock-based insertion (atomicCAS on child slots) the
// tree is derived from sorted keys, without locks (the only waits, bounded,
// are those of a sort or scan tile for the counts of the tiles before it):
//   1. per-instance bounding box -> root cube (lower corner = per-axis min,
//      edge s0 = max extent * (1 + 2^-20));
//   2. key = instance bits | Morton interleave of the cell index
//      k = floor((x - min) / s0 * 2^B) (B bits per axis);
//   3. stable sort of (key, particle) pairs: LSD radix, 8-bit digits, a launch
//      each; up to 16k pairs by counting, in one launch;
//   4. every slot i that starts a cell at some level emits that cell as a
//      node if its parent cell holds more than L particles; slot order then
//      level order is exactly pre-order, so the subtree of a node is the
//      contiguous id range [id, skip[id]) and walks need no stack;
//   5. node mass, centre of mass and tight box bottom-up: the last child to
//      arrive (atomic counter) combines its siblings in child order, so the
//      result does not depend on arrival order.
#include <climits>

#include "sph_internal.cuh"
#include "fpbits.cuh"
#include "morton.cuh"
#include "pack.cuh"

namespace sph {

// ---------------------------------------------------------------------------
// Bounding boxes and validity
// ---------------------------------------------------------------------------
// Words of Tree::look: counters and tickets, the digit histograms of the
// sort, then the look-back states of the sort's tiles and of the two scans.
enum { LK_BBOX = 0, LK_NODES, LK_GROUPS, LK_SORT = 8, LK_HIST = 64 };
constexpr int kLookFixed = LK_HIST + 8 * 256;

// Everything a build starts from, in one launch: the words of Tree::look it
// will use, the bounding boxes, no roots, no leaves.
__global__ void k_tree_init(Tree T, int64_t words, int ninst) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = t; i < words; i += step) T.look[i] = 0;
  for (int64_t i = t; i < ninst; i += step) {
    for (int ax = 0; ax < 3; ++ax) {
      T.inst_bb[6 * i + ax] = dbl_to_ord(__longlong_as_double(0x7ff0000000000000LL));  // +inf
      T.inst_bb[6 * i + 3 + ax] = dbl_to_ord(__longlong_as_double((long long)0xfff0000000000000ULL));  // -inf
    }
    T.inst_root[i] = -1;
  }
  if (t == 0) *T.nleaf = 0;
}

// min / max of order-preserving encodings (integer pipe)
__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v) {
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w < v ? w : v;
  }
  return v;
}
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  return v;
}

// Root cube per instance (Sect. 3.5.1): corner = per-axis minimum, edge
// s0 = max over axes of the extent, enlarged by 2^-20 so that the particle
// at the maximum falls inside; a zero extent (one particle) gives s0 = 1.
__device__ void make_root(const unsigned long long *bb, int i, int dim, double *lo_out, double *s0_out,
                          double *rs0_out) {
  double ext = 0.0;
  for (int ax = 0; ax < 3; ++ax) {
    double lo = ord_to_dbl(__ldcg(&bb[6 * i + ax])), hi = ord_to_dbl(__ldcg(&bb[6 * i + 3 + ax]));
    if (ax >= dim || !(hi >= lo)) {  // unused axis or empty instance
      lo = 0.0;
      hi = 0.0;
    }
    lo_out[3 * i + ax] = lo;
    ext = fmax(ext, __dsub_rn(hi, lo));
  }
  double s0 = __dmul_rn(ext, 1.0 + 0x1p-20);
  s0 = s0 > 0.0 ? s0 : 1.0;
  s0_out[i] = s0;
  rs0_out[i] = __drcp_rn(s0);
}

// Code units from particle 0 (see Units).
__device__ __forceinline__ double pow2_floor(double v) { return (v > 0.0 && isfinite(v)) ? ldexp(1.0, ilogb(v)) : 1.0; }

__device__ void make_units(const double *__restrict__ h, const double *__restrict__ m, int64_t n, int dim,
                           double vscale, const MatTable &mt, Units *U) {
  // every lane forms the (power-of-two) base units; lane i converts material i
  const double L = pow2_floor(n > 0 ? h[0] : 1.0), M = pow2_floor(n > 0 ? m[0] : 1.0);
  const double T = pow2_floor(L / (vscale > 0.0 ? vscale : 1.0));
  Units u;
  u.L = L;
  u.M = M;
  u.T = T;
  u.invL = 1.0 / L;
  u.invM = 1.0 / M;
  u.invT = 1.0 / T;
  u.rho = dim == 3 ? M / (L * L * L) : M / (L * L);  // density: mass per L^D
  u.invrho = 1.0 / u.rho;
  u.V = L / T;
  u.invV = 1.0 / u.V;
  u.sig = dim == 3 ? M / (L * T * T) : M / (T * T);  // stress: rho V^2
  u.invsig = 1.0 / u.sig;
  u.E = u.V * u.V;
  u.invE = 1.0 / u.E;
  u.acc = L / (T * T);
  u.Gs = 0.0;
  const int i = threadIdx.x;
  if (i < SPH_MAX_MATERIALS) {
    const sph_material &a = mt.m[i < mt.nmat ? i : 0];
    float *f = U->matf[i];
    f[MF_RHO0] = (float)(a.rho0 * u.invrho);
    f[MF_CS] = (float)(a.cs * u.invV);
    f[MF_K0] = (float)(a.K0 * u.invsig);
    f[MF_NM] = (float)a.n_M;
    f[MF_AT] = (float)(a.A_T * u.invsig);
    f[MF_BT] = (float)(a.B_T * u.invsig);
    f[MF_E0] = (float)(a.E0 * u.invE);
    f[MF_EIV] = (float)(a.E_iv * u.invE);
    f[MF_ECV] = (float)(a.E_cv * u.invE);
    f[MF_AA] = (float)a.a_T;
    f[MF_BB] = (float)a.b_T;
    f[MF_ALPHA] = (float)a.alpha_T;
    f[MF_BETA] = (float)a.beta_T;
    f[MF_RHOCUT] = (float)a.rho_cut;
    f[MF_MU] = (float)(a.mu * u.invsig);
    f[MF_Y0] = (float)(a.Y0 * u.invsig);
  }
  if (threadIdx.x == 0) {
    // base fields only: the material rows are written by their lanes
    U->L = u.L;
    U->M = u.M;
    U->T = u.T;
    U->invL = u.invL;
    U->invM = u.invM;
    U->invT = u.invT;
    U->rho = u.rho;
    U->invrho = u.invrho;
    U->V = u.V;
    U->invV = u.invV;
    U->sig = u.sig;
    U->invsig = u.invsig;
    U->E = u.E;
    U->invE = u.invE;
    U->acc = u.acc;
    U->Gs = u.Gs;
  }
}

// Bounding boxes: block (inst, j) takes chunks j, j + gridDim.y - 1, ... of
// its instance (one block per instance took 0.49 ms for 64 instances of up to
// 50k particles, now 0.04).  Also flags non-finite positions/velocities and h, rho that are
// not positive.  The block after the last column forms the code units
// meanwhile, and the last block to finish the root cubes.
struct BboxArgs {
  const double *x[3], *v[3], *h, *m, *rho;
  int64_t n;
  int dim, ninst;
  const int64_t *inst_off;
  double vscale;
  MatTable mt;
  Units *U;
  int32_t *err;
};
__global__ void __launch_bounds__(256) k_bbox(BboxArgs A, Tree T) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (blockIdx.y == gridDim.y - 1) {
    if (blockIdx.x == 0 && w == 0) make_units(A.h, A.m, A.n, A.dim, A.vscale, A.mt, A.U);
    return;
  }
  const int cols = gridDim.y - 1, inst = blockIdx.x, dim = A.dim;
  // extrema as order-preserving integers: comparisons stay off the FP64 unit
  unsigned long long lo[3] = {~0ULL, ~0ULL, ~0ULL}, hi[3] = {0ULL, 0ULL, 0ULL};
  const bool many = A.ninst > 1 && A.inst_off;
  const int64_t i0 = (many ? A.inst_off[inst] : 0) + (int64_t)blockIdx.y * blockDim.x + threadIdx.x;
  const int64_t i1 = many ? A.inst_off[inst + 1] : A.n, stride = (int64_t)cols * blockDim.x;
  bool bad = false;
  for (int64_t i = i0; i < i1; i += stride) {
    const double p[3] = {A.x[0][i], A.x[1][i], dim == 3 ? A.x[2][i] : 0.0};
    bad |= !finite_bits(p[0]) || !finite_bits(p[1]) || !finite_bits(p[2]) || !finite_bits(A.v[0][i]) ||
           !finite_bits(A.v[1][i]) || (dim == 3 && !finite_bits(A.v[2][i])) || !positive_finite_bits(A.h[i]) ||
           !positive_finite_bits(A.rho[i]);
    for (int ax = 0; ax < 3; ++ax) {
      const unsigned long long o = ord_of(p[ax]);
      lo[ax] = o < lo[ax] ? o : lo[ax];
      hi[ax] = o > hi[ax] ? o : hi[ax];
    }
  }
  if (bad) raise_err(A.err, ERR_NONFINITE);
  __shared__ unsigned long long s[6][32];
  __shared__ bool last;
  for (int ax = 0; ax < 3; ++ax) {
    unsigned long long a = warp_min_u64(lo[ax]), b = warp_max_u64(hi[ax]);
    if (lane == 0) {
      s[ax][w] = a;
      s[3 + ax][w] = b;
    }
  }
  __syncthreads();
  if (w == 0) {
    for (int ax = 0; ax < 3; ++ax) {
      unsigned long long a = lane < nw ? s[ax][lane] : ~0ULL;
      unsigned long long b = lane < nw ? s[3 + ax][lane] : 0ULL;
      a = warp_min_u64(a);
      b = warp_max_u64(b);
      if (lane == 0) {
        atomicMin(&T.inst_bb[6 * inst + ax], a);
        atomicMax(&T.inst_bb[6 * inst + 3 + ax], b);
      }
    }
    if (lane == 0) {
      __threadfence();
      last = atomicAdd(&T.look[LK_BBOX], 1u) == (uint32_t)cols * gridDim.x - 1u;
    }
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int i = threadIdx.x; i < A.ninst; i += blockDim.x)
    make_root(T.inst_bb, i, dim, T.inst_lo, T.inst_s0, T.inst_rs0);
}

// Morton keys, the histograms of all the digits the sort will use (a key's
// digits are the same in every pass) and, with `pack`, the FP32 views.  Both
// value buffers start as valid indices.
__global__ void __launch_bounds__(256) k_keys(const double *__restrict__ x, const double *__restrict__ y,
                                              const double *__restrict__ z, const double *__restrict__ vx,
                                              const double *__restrict__ vy, const double *__restrict__ vz,
                                              const double *__restrict__ h, const double *__restrict__ m,
                                              const double *__restrict__ rho, int64_t n, int dim, int B,
                                              const int64_t *__restrict__ inst_off, int ninst, int passes, bool pack,
                                              PackedF32 pk, const Units *__restrict__ U, Tree T) {
  __shared__ uint32_t hs[8][256];
  for (int p = 0; p < passes; ++p) hs[p][threadIdx.x] = 0;
  __syncthreads();
  const double *__restrict__ ilo = T.inst_lo;
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    const int inst = inst_of(inst_off, ninst, i);
    const double xa[3] = {x[i], y[i], dim == 3 ? z[i] : 0.0};
    const unsigned long long key = morton_key(xa, dim, B, inst, ilo, T.inst_s0[inst], T.inst_rs0[inst]);
    T.keys[0][i] = key;
    T.vals[0][i] = T.vals[1][i] = (int32_t)i;
    for (int p = 0; p < passes; ++p) atomicAdd(&hs[p][(key >> (8 * p)) & 255], 1u);
    if (pack)
      pack_particle(pk, i, dim, xa[0], xa[1], xa[2], vx[i], vy[i], dim == 3 ? vz[i] : 0.0, h[i], m[i], rho[i],
                    ilo + 3 * inst, U);
  }
  __syncthreads();
  for (int p = 0; p < passes; ++p)
    if (const uint32_t c = hs[p][threadIdx.x]) atomicAdd(&T.look[LK_HIST + 256 * p + threadIdx.x], c);
}

// FP32 views of the state (see PackedF32), in code units.
__global__ void k_pack(const double *__restrict__ x, const double *__restrict__ y, const double *__restrict__ z,
                       const double *__restrict__ vx, const double *__restrict__ vy, const double *__restrict__ vz,
                       const double *__restrict__ h, const double *__restrict__ m, const double *__restrict__ rho,
                       int64_t n, int dim, const int64_t *__restrict__ inst_off, int ninst,
                       const double *__restrict__ ilo, const Units *__restrict__ U, PackedF32 pk) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int inst = inst_of(inst_off, ninst, i);
  pack_particle(pk, i, dim, x[i], y[i], dim == 3 ? z[i] : 0.0, vx[i], vy[i], dim == 3 ? vz[i] : 0.0, h[i], m[i],
                rho[i], ilo + 3 * inst, U);
}

// ---------------------------------------------------------------------------
// Decoupled look-back (Merrill and Garland, "Single-pass parallel prefix scan
// with decoupled look-back"): a tile publishes its own count, adds up the
// counts of the tiles before it until it meets one that already knows its
// inclusive sum, and publishes its own.  Tiles are numbered by a ticket in
// the order their blocks start, so a tile only ever waits for blocks that
// are running.  Every wait is bounded; one that runs out raises the timeout
// bit and goes on with the sum so far, which every later access tolerates.
// State word W (one store, one load): its two top bits are 1 = the tile's own
// count, 2 = inclusive, the rest the count.  32 bits hold 2^30 - 1: enough for
// the particles of a digit and for walk groups, and for nodes, whose sums stop
// there and so exceed any node capacity that fits the device (236 bytes a node).
// Counts of other things than particles (k_scan) take 64 bits.
// ---------------------------------------------------------------------------
template <class W>
struct Look {
  static constexpr int kShift = 8 * sizeof(W) - 2;
  static constexpr W kOwn = (W)1 << kShift, kIncl = (W)2 << kShift, kVal = kOwn - 1;
};
constexpr uint32_t kLookOwn = Look<uint32_t>::kOwn, kLookIncl = Look<uint32_t>::kIncl, kLookVal = Look<uint32_t>::kVal;
constexpr int kLookPolls = 1 << 22;

template <class W>
__device__ __forceinline__ W look_load(const W *p) {
  return *(const volatile W *)p;
}

// Sum of the tiles before `tile` for one counter; called by a whole warp,
// lane i reading the i-th tile back.  Publishes the inclusive sum.
template <class W>
__device__ __forceinline__ W look_back_warp(W *state, int tile, W own, int32_t *err) {
  using K = Look<W>;
  const int lane = threadIdx.x & 31;
  if (lane == 0) *(volatile W *)&state[tile] = own | (tile == 0 ? K::kIncl : K::kOwn);
  W before = 0;
  for (int t = tile - 1; t >= 0; t -= 32) {
    const int mine = t - lane;
    W v = K::kIncl;  // before the first tile: nothing, known
    if (mine >= 0) {
      int polls = 0;
      while (((v = look_load(&state[mine])) >> K::kShift) == 0 && ++polls < kLookPolls) __nanosleep(20);
      if (polls >= kLookPolls) raise_err(err, ERR_TIMEOUT);
    }
    const unsigned incl = __ballot_sync(0xffffffffu, (v >> K::kShift) != 1);
    const int last = incl ? __ffs(incl) - 1 : 31;
    W sum = lane <= last ? v & K::kVal : (W)0;
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    before = min(before + sum, (W)K::kVal);
    if (incl) break;
  }
  if (lane == 0 && tile > 0) *(volatile W *)&state[tile] = min(before + own, (W)K::kVal) | K::kIncl;
  return before;
}

template <class T>
__device__ __forceinline__ T block_excl_scan(T v, T *total) {
  __shared__ T ws[32];
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  T s = v;
  for (int o = 1; o < 32; o <<= 1) {
    T t = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += t;
  }
  if (lane == 31) ws[w] = s;
  __syncthreads();
  if (w == 0) {
    T t = lane < nw ? ws[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      T u = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += u;
    }
    ws[lane] = t;
  }
  __syncthreads();
  T res = s - v + (w > 0 ? ws[w - 1] : 0);
  *total = ws[nw - 1];
  __syncthreads();
  return res;
}

// ---------------------------------------------------------------------------
// LSD radix sort of (u64 key, i32 value), 8-bit digits, stable: one launch per
// digit, each reading and writing its pairs once ("onesweep", Adinets and
// Merrill).  The digit totals come from one histogram pass over the keys.  A
// tile ranks its pairs by warp matching, looks back per digit (a thread per
// digit, eight tiles at a time) and scatters.  The histogram, three scan
// kernels and scatter per digit that this replaces took 311 us of a 1M build
// and 163 of a 4.4k one, nearly all of the latter latency; now 212 and 48 us.
// ---------------------------------------------------------------------------
constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kLookWin = 8;
constexpr int kSortWarps = kSortThreads / 32;

__global__ void __launch_bounds__(kSortThreads) k_sort_hist(const unsigned long long *__restrict__ keys, int64_t n,
                                                            int passes, uint32_t *hist) {
  __shared__ uint32_t hs[8][256];
  for (int p = 0; p < passes; ++p) hs[p][threadIdx.x] = 0;
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * kSortThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kSortThreads) {
    const unsigned long long k = keys[i];
    for (int p = 0; p < passes; ++p) atomicAdd(&hs[p][(k >> (8 * p)) & 255], 1u);
  }
  __syncthreads();
  for (int p = 0; p < passes; ++p)
    if (const uint32_t c = hs[p][threadIdx.x]) atomicAdd(&hist[256 * p + threadIdx.x], c);
}

__global__ void __launch_bounds__(kSortThreads) k_sort_pass(const unsigned long long *__restrict__ kin,
                                                            const int32_t *__restrict__ vin,
                                                            unsigned long long *__restrict__ kout,
                                                            int32_t *__restrict__ vout, int64_t n, int shift,
                                                            const uint32_t *__restrict__ hist, uint32_t *state,
                                                            uint32_t *ticket, int32_t *err) {
  __shared__ uint32_t wc[kSortWarps][256];
  __shared__ uint32_t base[256];
  __shared__ int tile_s;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, t = threadIdx.x;
  const unsigned lt = (1u << lane) - 1u;
  if (t == 0) tile_s = (int)atomicAdd(ticket, 1u);
#pragma unroll
  for (int ww = 0; ww < kSortWarps; ++ww) wc[ww][t] = 0;
  __syncthreads();
  const int tile = tile_s;
  // a warp's pairs are consecutive, so that rank order is input order
  const int64_t first = (int64_t)tile * kSortTile + w * (32 * kSortItems) + lane;
  unsigned long long key[kSortItems];
  int32_t val[kSortItems];
  uint32_t rank[kSortItems];
#pragma unroll
  for (int j = 0; j < kSortItems; ++j) {
    const int64_t i = first + 32 * j;
    key[j] = i < n ? kin[i] : 0ULL;
    val[j] = i < n ? vin[i] : 0;
  }
#pragma unroll
  for (int j = 0; j < kSortItems; ++j) {
    const bool valid = first + 32 * j < n;
    const int d = valid ? (int)((key[j] >> shift) & 255) : 256;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const int leader = __ffs(peers) - 1;
    uint32_t before = 0;
    if (valid && lane == leader) {
      before = wc[w][d];
      wc[w][d] = before + __popc(peers);
    }
    rank[j] = __shfl_sync(0xffffffffu, before, leader) + __popc(peers & lt);
    __syncwarp();
  }
  __syncthreads();
  // thread t: digit t
  uint32_t own = 0;
#pragma unroll
  for (int ww = 0; ww < kSortWarps; ++ww) {
    const uint32_t c = wc[ww][t];
    wc[ww][t] = own;
    own += c;
  }
  volatile uint32_t *mine = state + (int64_t)tile * 256 + t;
  *mine = own | (tile == 0 ? kLookIncl : kLookOwn);
  uint32_t before = 0;
  bool known = tile == 0;
  for (int q = tile - 1; q >= 0 && !known; q -= kLookWin) {
    uint32_t v[kLookWin];
#pragma unroll
    for (int u = 0; u < kLookWin; ++u) v[u] = q - u >= 0 ? look_load(&state[(int64_t)(q - u) * 256 + t]) : kLookIncl;
#pragma unroll
    for (int u = 0; u < kLookWin; ++u) {
      if (known) continue;
      int polls = 0;
      while ((v[u] >> 30) == 0u && ++polls < kLookPolls) {
        __nanosleep(20);
        v[u] = look_load(&state[(int64_t)(q - u) * 256 + t]);
      }
      if (polls >= kLookPolls) raise_err(err, ERR_TIMEOUT);
      before += v[u] & kLookVal;
      known = (v[u] >> 30) != 1u;
    }
  }
  if (tile > 0) *mine = (before + own) | kLookIncl;
  int32_t total;
  base[t] = (uint32_t)block_excl_scan((int32_t)hist[t], &total) + before;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kSortItems; ++j) {
    if (first + 32 * j >= n) continue;
    const int d = (int)((key[j] >> shift) & 255);
    const int64_t pos = (int64_t)base[d] + wc[w][d] + rank[j];
    if (pos < n) {
      kout[pos] = key[j];
      vout[pos] = val[j];
    }
  }
}

// The same sort for n <= kSmallSort in one launch: a pair's place is the number
// of pairs before it in (key, index) order, counted against every key.  A
// block places 32 pairs, a lane each; its warps share out the keys, read from
// shared memory two at a time.  n^2 comparisons of about four instructions over
// the whole chip, against a launch per digit with a few tiles at 7.5 us each.
// A 3D tree and partner lists, with and without it: 4.1k particles 279 / 349 us,
// 8.0k 289 / 354, 13.9k 316 / 353, 22k 385 / 371, 33k 512 / 400; so the line is
// drawn at 16k.  (The digits in one block's shared memory: 39 us for six digits
// of 4.4k keys, against 6 us here.)
constexpr int kRankThreads = 512, kRankTile = 2048;
constexpr int64_t kSmallSort = 16384;

__global__ void __launch_bounds__(kRankThreads) k_sort_small(const unsigned long long *__restrict__ kin,
                                                             const int32_t *__restrict__ vin,
                                                             unsigned long long *__restrict__ kout,
                                                             int32_t *__restrict__ vout, int n) {
  constexpr int W = kRankThreads / 32;
  __shared__ __align__(16) unsigned long long sk[kRankTile];
  __shared__ int red[W][32];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int i0 = blockIdx.x * 32, i = i0 + lane;
  const unsigned long long ki = i < n ? kin[i] : 0ULL;
  int cnt = 0;
  for (int j0 = 0; j0 < n; j0 += kRankTile) {
    const int m = min(kRankTile, n - j0), share = ((m + 2 * W - 1) / (2 * W)) * 2;
    __syncthreads();
    // past the end: a key that counts for none (m is odd only when n - j0 is)
    for (int k = t; k < ((m + 1) & ~1); k += kRankThreads) sk[k] = k < m ? kin[j0 + k] : ~0ULL;
    __syncthreads();
    const int a = min(w * share, (m + 1) & ~1), b = min(a + share, (m + 1) & ~1);
    // keys before the block's own pairs, among them, after them
    const int own = min(max(i0 - j0, a), b), past = min(max(i0 + 32 - j0, a), b);
    const ulonglong2 *s2 = (const ulonglong2 *)sk;
#pragma unroll 8
    for (int k = a; k < own; k += 2) {
      const ulonglong2 q = s2[k >> 1];
      cnt += q.x <= ki ? 1 : 0;
      cnt += q.y <= ki ? 1 : 0;
    }
    for (int k = own; k < past; ++k) cnt += (sk[k] < ki || (sk[k] == ki && j0 + k < i)) ? 1 : 0;
#pragma unroll 8
    for (int k = past; k < b; k += 2) {
      const ulonglong2 q = s2[k >> 1];
      cnt += q.x < ki ? 1 : 0;
      cnt += q.y < ki ? 1 : 0;
    }
  }
  red[w][lane] = cnt;
  __syncthreads();
  if (w > 0 || i >= n) return;
  int pos = 0;
#pragma unroll
  for (int k = 0; k < W; ++k) pos += red[k][lane];
  kout[pos] = ki;
  vout[pos] = vin[i];
}

static int sort_passes(int bits) { return (bits + 7) / 8; }

// The passes; above kSmallSort with Tree::look zeroed and its histograms filled
static void sort_run(sph_ctx *c, int64_t n, int bits, cudaStream_t st) {
  Tree &T = c->tree;
  const int tiles = nblk(n, kSortTile), passes = sort_passes(bits);
  if (n <= kSmallSort) {
    { k_sort_small<<<nblk(n, 32), kRankThreads, 0, st>>>(T.keys[0], T.vals[0], T.keys[1], T.vals[1], (int)n); ++sph::g_launches; }
    T.skey = T.keys[1];
    T.perm = T.vals[1];
    return;
  }
  int src = 0;
  for (int p = 0; p < passes; ++p) {
    k_sort_pass<<<tiles, kSortThreads, 0, st>>>(T.keys[src], T.vals[src], T.keys[src ^ 1], T.vals[src ^ 1], n, 8 * p,
                                                T.look + LK_HIST + 256 * p,
                                                T.look + kLookFixed + (int64_t)p * tiles * 256, T.look + LK_SORT + p,
                                                c->d_err);
    ++sph::g_launches;
    src ^= 1;
  }
  T.skey = T.keys[src];
  T.perm = T.vals[src];
}

// Sorts (keys[0], vals[0]) of the tree's sort buffers; the result is left
// in (skey, perm).  Used outside the tree build by the flaw generator and the
// fragment finder, which do not need the tree afterwards.
void sort_pairs(sph_ctx *c, int64_t n, int bits, cudaStream_t st) {
  Tree &T = c->tree;
  if (n <= 0) {
    T.skey = T.keys[0];
    T.perm = T.vals[0];
    return;
  }
  if (n <= kSmallSort) {
    sort_run(c, n, bits, st);
    return;
  }
  const int passes = sort_passes(bits);
  cudaMemsetAsync(T.look, 0, sizeof(uint32_t) * (kLookFixed + (int64_t)passes * nblk(n, kSortTile) * 256), st);
  k_sort_hist<<<std::min(nblk(n, kSortThreads), 2 * c->num_sms), kSortThreads, 0, st>>>(T.keys[0], n, passes,
                                                                                       T.look + LK_HIST);
  ++sph::g_launches;
  sort_run(c, n, bits, st);
}

// ---------------------------------------------------------------------------
// Exclusive scan of non-negative int32 counts (length m), one pass.  Sums are
// kept in 64 bits (partners and flaws number more than 2^30 well within the
// device's memory); O holds the offsets.
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 256, kScanItems = 16, kScanTile = kScanThreads * kScanItems;

template <class O>
__global__ void __launch_bounds__(kScanThreads) k_scan(const int32_t *in, O *out,  // may be the same
                                                       int64_t m, uint32_t *ticket, uint64_t *state, int32_t *err) {
  __shared__ int tile_s;
  __shared__ uint64_t before_s;
  if (threadIdx.x == 0) tile_s = (int)atomicAdd(ticket, 1u);
  __syncthreads();
  const int64_t at = (int64_t)tile_s * kScanTile + (int64_t)threadIdx.x * kScanItems;
  int32_t v[kScanItems];
  int64_t s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    v[k] = (at + k < m) ? in[at + k] : 0;
    s += v[k];
  }
  int64_t tot;
  int64_t off = block_excl_scan(s, &tot);
  if (threadIdx.x < 32) {
    const uint64_t b = look_back_warp(state, tile_s, (uint64_t)tot, err);
    if (threadIdx.x == 0) before_s = b;
  }
  __syncthreads();
  off += (int64_t)before_s;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    if (at + k < m) out[at + k] = (O)off;
    off += v[k];
  }
}

template <class O>
static void scan_run(sph_ctx *c, const int32_t *in, O *out, int64_t m, cudaStream_t st) {
  static_assert(kLookFixed % 2 == 0, "64-bit state words");
  Tree &T = c->tree;
  const int tiles = nblk(m, kScanTile);
  cudaMemsetAsync(T.look, 0, sizeof(uint32_t) * (kLookFixed + 2 * (int64_t)tiles), st);
  k_scan<<<tiles, kScanThreads, 0, st>>>(in, out, m, T.look, (uint64_t *)(T.look + kLookFixed), c->d_err);
  ++sph::g_launches;
}
// 32-bit offsets: the caller's total is at most 2^31 - 1
void scan_counts(sph_ctx *c, const int32_t *in, int32_t *out, int64_t m, cudaStream_t st) {
  scan_run(c, in, out, m, st);
}
void scan_counts(sph_ctx *c, const int32_t *in, int64_t *out, int64_t m, cudaStream_t st) {
  scan_run(c, in, out, m, st);
}

// Words of Tree::look a context for N particles and `cap` nodes needs: a
// build's sort and its two scans (or any other sort or scan alone).
int64_t look_words(int64_t N, int64_t cap) {
  return kLookFixed + (int64_t)8 * 256 * ((N + kSortTile - 1) / kSortTile) + (N + 256) / 256 + (cap + 255) / 256 + 8;
}

// ---------------------------------------------------------------------------
// Node emission
// ---------------------------------------------------------------------------
struct KeyLevels {
  const unsigned long long *key;
  int dim, B;
  __device__ __forceinline__ unsigned long long prefix(int64_t i, int l) const { return key[i] >> (dim * (B - l)); }
  // deepest level at which two slots (i-1 and i) share a cell; -1 if they lie
  // in different instances
  __device__ __forceinline__ int common(int64_t i) const { return shared(i - 1, i); }
  __device__ __forceinline__ int shared(int64_t i, int64_t j) const {
    unsigned long long d = key[i] ^ key[j];
    if (d == 0) return B;
    int hb = 63 - __clzll((long long)d);
    if (hb >= dim * B) return -1;
    return B - 1 - hb / dim;
  }
  // first slot in [lo, hi) whose level-l prefix exceeds p
  __device__ __forceinline__ int64_t upper(unsigned long long p, int l, int64_t lo, int64_t hi) const {
    while (lo < hi) {
      int64_t mid = (lo + hi) >> 1;
      if (prefix(mid, l) <= p) lo = mid + 1; else hi = mid;
    }
    return lo;
  }
  // first slot in [lo, hi) whose level-l prefix is >= p
  __device__ __forceinline__ int64_t lower(unsigned long long p, int l, int64_t lo, int64_t hi) const {
    while (lo < hi) {
      int64_t mid = (lo + hi) >> 1;
      if (prefix(mid, l) < p) lo = mid + 1; else hi = mid;
    }
    return lo;
  }
  // Deepest level at which the cell that starts at slot i holds more than L
  // particles, or -1: the keys are sorted, so it holds slot i + L as well.
  __device__ __forceinline__ int split_level(int64_t i, int L, int64_t n) const {
    return i + L < n ? shared(i, i + L) : -1;
  }
};

__device__ __forceinline__ void slot_segment(const int64_t *inst_off, int ninst, int64_t n, int64_t i, int64_t &lo,
                                             int64_t &hi) {
  if (ninst > 1 && inst_off) {
    int k = inst_of(inst_off, ninst, i);
    lo = inst_off[k];
    hi = inst_off[k + 1];
  } else {
    lo = 0;
    hi = n;
  }
}

// First level at which slot i starts a cell that is a node, or B+1 if none;
// `split` is its split_level where that is at hand, else -1.
__device__ __forceinline__ int first_node_level(const KeyLevels &K, int64_t i, int64_t seg_lo, int64_t seg_hi,
                                                int L, int split) {
  int c = (i == seg_lo) ? -1 : K.common(i);
  int l0 = c + 1;
  if (l0 > K.B) return K.B + 1;
  if (l0 > 0 && split < l0 - 1) {
    unsigned long long pp = K.prefix(i, l0 - 1);
    int64_t lo = K.lower(pp, l0 - 1, max(seg_lo, i - L), i);
    int64_t hi = K.upper(pp, l0 - 1, i + 1, min(seg_hi, i + L + 1));
    if (hi - lo <= L) return K.B + 1;  // the parent cell is a leaf (or lies below one)
  }
  return l0;
}

// Nodes that start at each slot, and their scan (nstart[n] = their number); a
// slot's nodes also get their children and arrival counts cleared.  A slot's
// nodes are the levels from its first to the first that does not split, which
// one comparison of keys L slots apart tells: searching each cell's end took
// 11 us for 4.4k particles (now 5.6), 71 us for 1M (now 43).
// IT slots per thread: four shorten the look-back's chain of tiles, at small n
// one spreads the slots over more SMs.  One, four, eight: a tree and partner
// lists of 4.1k particles 272, 275, 283 us, 33k 397, 396, 400, 111k 528, 523,
// 527, 263k 794, 786, 790; the mixed adjoint at 1M 4452, 4426, 4437 us.
template <int IT>
__global__ void __launch_bounds__(256) k_node_scan(KeyLevels K, int64_t n, int L, const int64_t *__restrict__ inst_off,
                                                   int ninst, Tree T, uint32_t *state, int32_t *err) {
  __shared__ int tile_s;
  __shared__ uint32_t before_s;
  if (threadIdx.x == 0) tile_s = (int)atomicAdd(&T.look[LK_NODES], 1u);
  __syncthreads();
  const int64_t first = ((int64_t)tile_s * 256 + threadIdx.x) * IT;
  int nodes[IT], sum = 0;
#pragma unroll
  for (int j = 0; j < IT; ++j) {
    const int64_t i = first + j;
    nodes[j] = 0;
    if (i < n) {
      int64_t seg_lo, seg_hi;
      slot_segment(inst_off, ninst, n, i, seg_lo, seg_hi);
      const int split = K.split_level(i, L, n), l0 = first_node_level(K, i, seg_lo, seg_hi, L, split);
      if (l0 <= K.B) nodes[j] = min(max(l0, split + 1), K.B) - l0 + 1;
    }
    sum += nodes[j];
  }
  int32_t tot;
  int32_t off = block_excl_scan(sum, &tot);
  if (threadIdx.x < 32) {
    const uint32_t b = look_back_warp(state, tile_s, (uint32_t)tot, err);
    if (threadIdx.x == 0) before_s = b;
  }
  __syncthreads();
  off += (int32_t)before_s;
  int4 *child = reinterpret_cast<int4 *>(T.child);
#pragma unroll
  for (int j = 0; j < IT; ++j) {
    const int64_t i = first + j;
    if (i > n) return;
    T.nstart[i] = off;
    if (i == n) {
      *T.nnodes = off <= T.cap_nodes ? off : (int32_t)T.cap_nodes;
      if (off > T.cap_nodes) raise_err(err, ERR_NODE_OVERFLOW);
      return;
    }
    for (int64_t id = off; id < off + nodes[j] && id < T.cap_nodes; ++id) {
      T.nchild[id] = T.arrived[id] = 0;
      child[2 * id] = child[2 * id + 1] = make_int4(-1, -1, -1, -1);
    }
    off += nodes[j];
  }
}

__global__ void k_node_emit(KeyLevels K, int64_t n, int L, const int64_t *__restrict__ inst_off, int ninst,
                            const int32_t *__restrict__ nstart, Tree T) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || nstart[i + 1] == nstart[i]) return;
  int64_t seg_lo, seg_hi;
  slot_segment(inst_off, ninst, n, i, seg_lo, seg_hi);
  if (i == seg_lo) T.inst_root[inst_of(inst_off, ninst, i)] = nstart[i];
  int l0 = first_node_level(K, i, seg_lo, seg_hi, L, -1);
  int32_t parent = -1;
  if (l0 > 0) {
    // the parent cell starts at slot p; its node is the (l0-1 - l0(p))-th of p's chain
    unsigned long long pp = K.prefix(i, l0 - 1);
    int64_t p = K.lower(pp, l0 - 1, seg_lo, i);
    int lp = (p == seg_lo) ? 0 : K.common(p) + 1;
    parent = nstart[p] + (l0 - 1 - lp);
  }
  int64_t e = seg_hi;
  int32_t id = nstart[i];
  for (int l = l0; l <= K.B; ++l, ++id) {
    int64_t end = K.upper(K.prefix(i, l), l, i + 1, e);
    if (id < T.cap_nodes) {
      T.first[id] = (int32_t)i;
      T.end[id] = (int32_t)end;
      T.level[id] = l;
      T.cell[id] = K.prefix(i, l);
      T.skip[id] = min((int64_t)nstart[end], T.cap_nodes);
      T.nrec[id] = make_int4((int32_t)i, (int32_t)end, T.skip[id], l);
      T.parent[id] = parent;
      if (parent >= 0 && parent < id) {  // a parent always comes first
        atomicAdd(&T.nchild[parent], 1);
        T.child[8 * (int64_t)parent + (int)(K.prefix(i, l) & ((1u << K.dim) - 1u))] = id;
      }
    }
    parent = id;
    if (end - i <= L || l == K.B) break;
    e = end;
  }
  // the chain ends at a leaf: list it for the moments pass
  if (id < T.cap_nodes) {
    const unsigned mask = __activemask();
    const int lane = threadIdx.x & 31, leader = __ffs(mask) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(T.nleaf, __popc(mask));
    base = __shfl_sync(mask, base, leader);
    T.ncount[base + __popc(mask & ((1u << lane) - 1u))] = id;
  }
}

// Walk groups: runs of consecutive sibling cells that each hold at most 32
// particles, packed greedily up to 32 particles by their parent (a node with
// more than 32); a root with at most 32 particles is one group, and a leaf at
// full depth with more than 32 is cut into runs of 32.  Siblings are adjacent
// in Morton order, so a group is a compact block of space, and together the
// groups partition the particles in slot order.
__device__ __forceinline__ int node_count(const Tree &T, int32_t id) { return T.end[id] - T.first[id]; }

template <bool EMIT>
__device__ int group_runs(const Tree &T, int32_t id, int32_t g0, int inst) {
  const int c = node_count(T, id);
  const bool leaf = c <= T.leaf_size || T.level[id] == T.max_depth;
  int g = 0;
  if (c <= kWarp) {
    if (T.parent[id] >= 0) return 0;  // packed by its parent
    if (EMIT && g0 < T.cap_groups) {
      T.grp_start[g0] = T.first[id];
      T.grp_end[g0] = T.end[id];
      T.grp_inst[g0] = inst;
    }
    return 1;
  }
  if (leaf) {
    const int32_t f = T.first[id], e = T.end[id];
    for (int32_t s = f; s < e; s += kWarp, ++g)
      if (EMIT && g0 + g < T.cap_groups) {
        T.grp_start[g0 + g] = s;
        T.grp_end[g0 + g] = min(s + kWarp, e);
        T.grp_inst[g0 + g] = inst;
      }
    return g;
  }
  int32_t run_s = -1, run_e = -1;
  int run = 0;
  const int32_t stop = T.skip[id];
  int guard = 0;
  for (int32_t ch = id + 1; ch < stop && guard < 64; ch = T.skip[ch], ++guard) {
    const int cc = node_count(T, ch);
    if (cc <= kWarp && run + cc <= kWarp) {
      if (run == 0) run_s = T.first[ch];
      run += cc;
      run_e = T.end[ch];
      continue;
    }
    if (run > 0) {  // close the current run
      if (EMIT && g0 + g < T.cap_groups) {
        T.grp_start[g0 + g] = run_s;
        T.grp_end[g0 + g] = run_e;
        T.grp_inst[g0 + g] = inst;
      }
      ++g;
      run = 0;
    }
    if (cc <= kWarp) {  // starts a new run
      run_s = T.first[ch];
      run_e = T.end[ch];
      run = cc;
    }
  }
  if (run > 0) {
    if (EMIT && g0 + g < T.cap_groups) {
      T.grp_start[g0 + g] = run_s;
      T.grp_end[g0 + g] = run_e;
      T.grp_inst[g0 + g] = inst;
    }
    ++g;
  }
  return g;
}

// Counts a node's groups, scans the counts and writes the groups, in tiles of
// 256 nodes (the number of nodes is only known on the device: the resident
// blocks draw tiles until there are none).
__global__ void __launch_bounds__(256) k_groups(Tree T, const int64_t *__restrict__ inst_off, int ninst,
                                                uint32_t *state, int32_t *err) {
  __shared__ int tile_s;
  __shared__ uint32_t before_s;
  const int nn = *T.nnodes, tiles = max(1, (nn + 255) / 256);
  for (;;) {
    if (threadIdx.x == 0) tile_s = (int)atomicAdd(&T.look[LK_GROUPS], 1u);
    __syncthreads();
    const int tile = tile_s;
    if (tile >= tiles) return;
    const int64_t id = (int64_t)tile * 256 + threadIdx.x;
    const int k = id < nn ? group_runs<false>(T, (int32_t)id, 0, 0) : 0;
    int32_t tot;
    int32_t off = block_excl_scan(k, &tot);
    if (threadIdx.x < 32) {
      const uint32_t b = look_back_warp(state, tile, (uint32_t)tot, err);
      if (threadIdx.x == 0) before_s = b;
    }
    __syncthreads();
    off += (int32_t)before_s;
    if (k > 0) group_runs<true>(T, (int32_t)id, off, inst_of(inst_off, ninst, T.first[id]));
    if (tile == tiles - 1 && threadIdx.x == 255) *T.ngroups = min(off + k, (int32_t)T.cap_groups);
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Node moments, bottom-up
// ---------------------------------------------------------------------------

// Bottom-up sums, eight lanes per node: mass, the mass-weighted position sum
// (kept in T.com until k_node_finish divides it), the particle box and h_max.  A
// warp takes four leaves, a lane every eighth particle; whoever arrives last
// at a parent combines its children, a lane per octant, four parents of the
// warp at a time.  Sums are taken over
// the lanes in a fixed order, so they are deterministic.  Extrema are kept as
// order-preserving integers and h_max as the bits of a positive double: only
// the sums use the FP64 unit.
// Bound by latency: a level costs a fence, an atomic and two dependent loads
// before its arithmetic.  With a thread per leaf, which loaded its particles
// one after the other and combined eight children by itself, a level of a 4.4k
// build took 6 us: 52 us in all, 117 at 263k, 180 at 1M, 320 at 2M; now 24, 56,
// 120 and 230 (8, 16 or 32 leaves a warp: the same at 1M, up to 8 % of a 4.4k
// step slower).
struct Moments {
  double M, mx[3];
  unsigned long long lo[3], hi[3], hm;
  __device__ __forceinline__ void clear() {
    M = 0.0;
    hm = 0ULL;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      mx[ax] = 0.0;
      lo[ax] = ~0ULL;
      hi[ax] = 0ULL;
    }
  }
  __device__ __forceinline__ void extrema(int ax, unsigned long long l, unsigned long long h) {
    lo[ax] = l < lo[ax] ? l : lo[ax];
    hi[ax] = h > hi[ax] ? h : hi[ax];
  }
  // over each eight lanes of `mask`
  template <int DIM>
  __device__ __forceinline__ void reduce(unsigned mask) {
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      M += __shfl_xor_sync(mask, M, o);
      const unsigned long long w = __shfl_xor_sync(mask, hm, o);
      hm = w > hm ? w : hm;
#pragma unroll
      for (int ax = 0; ax < DIM; ++ax) {
        mx[ax] += __shfl_xor_sync(mask, mx[ax], o);
        extrema(ax, __shfl_xor_sync(mask, lo[ax], o), __shfl_xor_sync(mask, hi[ax], o));
      }
    }
  }
  // lane `sub` of the team stores what falls to it
  template <int DIM>
  __device__ __forceinline__ void store(const Tree &T, int64_t node, int sub) const {
    const int64_t cap = T.cap_nodes;
    if (sub == 0) T.mass[node] = M;
    if (sub == 1) T.hmax[node] = bitsd(hm);
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      const bool use = ax < DIM;
      if (sub == 2 + ax) T.com[ax * cap + node] = use ? mx[ax] : 0.0;
      if (sub == 5 + ax) T.bblo[ax * cap + node] = use ? of_ord(lo[ax]) : 0.0;
      if (sub == (2 * ax + 2) % 8) T.bbhi[ax * cap + node] = use ? of_ord(hi[ax]) : 0.0;
    }
  }
};

template <int DIM>
__global__ void __launch_bounds__(128) k_moments(Tree T, const double *__restrict__ x, const double *__restrict__ y,
                                                 const double *__restrict__ z, const double *__restrict__ m,
                                                 const double *__restrict__ h) {
  const int lane = threadIdx.x & 31, sub = lane & 7, team = lane >> 3;
  const unsigned all = 0xffffffffu;
  const int64_t cap = T.cap_nodes;
  const double *X[3] = {x, y, z};
  const int nleaf = *T.nleaf;
  const int64_t l0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 4;
  if (l0 >= nleaf) return;
  const int32_t leaf = l0 + team < nleaf ? T.ncount[l0 + team] : -1;
  const int32_t end = leaf >= 0 ? T.end[leaf] : 0;
  Moments s;
  s.clear();
#pragma unroll 2
  for (int32_t j = (leaf >= 0 ? T.first[leaf] : 0) + sub; j < end; j += 8) {
    const int32_t a = T.perm[j];
    const double ma = m[a];
    const unsigned long long hb = dbits(h[a]);
    s.M += ma;
    s.hm = hb > s.hm ? hb : s.hm;
#pragma unroll
    for (int ax = 0; ax < DIM; ++ax) {
      const double v = X[ax][a];
      s.mx[ax] += ma * v;
      const unsigned long long o = ord_of(v);
      s.extrema(ax, o, o);
    }
  }
  __syncwarp();
  s.reduce<DIM>(all);
  if (leaf >= 0) s.store<DIM>(T, leaf, sub);
  int32_t node = sub == 0 ? leaf : -1;  // finished, its parent to be told by this lane
  // upwards: of the nodes finished in a round, those that complete a parent
  while (__any_sync(all, node >= 0)) {
    // the lane that counts up the parent fences after the warp's barrier, so
    // that the stores of all its team's lanes come before its count; the lanes
    // that read children likewise come after a barrier past the last one's fence
    __syncwarp();
    __threadfence();
    const int32_t p = node >= 0 ? T.parent[node] : -1;
    const bool win = p >= 0 && atomicAdd(&T.arrived[p], 1) == T.nchild[p] - 1;
    node = win ? p : -1;
    unsigned todo = __ballot_sync(all, win);
    if (todo) {
      __threadfence();
      __syncwarp();
    }
    while (todo) {
      unsigned pick = todo;  // team t takes the t-th parent left
      for (int t = 0; t < team; ++t) pick &= pick - 1;
      const int src = pick ? __ffs(pick) - 1 : 0;
      const int32_t q = __shfl_sync(all, p, src);
      const int32_t c = pick ? __ldcg(&T.child[8 * (int64_t)q + sub]) : -1;
      s.clear();
      if (c >= 0) {
        s.M = __ldcg(&T.mass[c]);
        s.hm = dbits(__ldcg(&T.hmax[c]));
#pragma unroll
        for (int ax = 0; ax < DIM; ++ax) {
          s.mx[ax] = __ldcg(&T.com[ax * cap + c]);
          s.lo[ax] = ord_of(__ldcg(&T.bblo[ax * cap + c]));
          s.hi[ax] = ord_of(__ldcg(&T.bbhi[ax * cap + c]));
        }
      }
      s.reduce<DIM>(all);
      if (pick) s.store<DIM>(T, q, sub);
      for (int t = 0; t < 4; ++t) todo &= todo - 1;
    }
  }
}

// Per node, all warps full: centre of mass from the sums, and the FP32 words
// of the walks in code units relative to the instance corner - the box rounded
// outwards with +-h_max (negative where the partner walk stops: at most
// max(L, walk_leaf) particles or depth B) and skip[], and the COM as hi + lo
// with the mass and the cell edge s0 / 2^level.
__global__ void k_node_finish(Tree T, int dim, int L, const int64_t *__restrict__ inst_off, int ninst,
                              const Units *__restrict__ U, int walk_leaf) {
  const int64_t node = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (node >= *T.nnodes) return;
  const int Lw = max(L, walk_leaf);
  const int64_t cap = T.cap_nodes;
  const int32_t nf = T.first[node], ne = T.end[node];
  const int inst = inst_of(inst_off, ninst, nf);
  const int kL = pow2_exp(U->invL), kM = pow2_exp(U->invM);
  const double M = T.mass[node], iM = 1.0 / M, hmax = T.hmax[node];
  float bl[3] = {0.f, 0.f, 0.f}, bh[3] = {0.f, 0.f, 0.f}, chi[3] = {0.f, 0.f, 0.f}, clo[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    if (ax >= dim) break;
    const double ilo = T.inst_lo[3 * inst + ax];
    const double com = T.com[ax * cap + node] * iM;
    T.com[ax * cap + node] = com;
    const double dl = __dsub_rn(T.bblo[ax * cap + node], ilo), dh = __dsub_rn(T.bbhi[ax * cap + node], ilo);
    bl[ax] = to_f32_dir_scaled(dl, kL, false, U->invL);
    bh[ax] = to_f32_dir_scaled(dh, kL, true, U->invL);
    to_f32_split_scaled(__dsub_rn(com, ilo), kL, U->invL, chi[ax], clo[ax]);
  }
  const float hf = to_f32_dir_scaled(hmax, kL, true, U->invL), mf = to_f32_scaled(M, kM, U->invM);
  const int lev = T.level[node];
  // edge s0 / 2^level: one exponent shift (the fallback's scale 2^(kL - level)
  // is built from its bits)
  const float ef = to_f32_scaled(T.inst_s0[inst], kL - lev, bitsd((uint64_t)(1023 + kL - lev) << 52));
  const bool stop = ne - nf <= Lw || lev == T.max_depth;
  // the gravity walk's word: skip, level and whether the walk sums the node's
  // members directly (its leaf test); the edge follows from the level
  const bool gleaf = ne - nf <= L || lev == T.max_depth;
  const float wf = T.packed_walk ? __uint_as_float((uint32_t)T.skip[node] | ((uint32_t)lev << 26) |
                                                   (gleaf ? 0x80000000u : 0u))
                                 : ef;
  T.fbox_lo[node] = make_float4(bl[0], bl[1], bl[2], stop ? -hf : hf);
  T.fbox_hi[node] = make_float4(bh[0], bh[1], bh[2], __int_as_float(T.skip[node]));
  T.fcom_hi[node] = make_float4(chi[0], chi[1], chi[2], mf);
  T.fcom_lo[node] = make_float4(clo[0], clo[1], clo[2], wf);
}

// ---------------------------------------------------------------------------
// Host orchestration
// ---------------------------------------------------------------------------
void pack_f32(sph_ctx *c, const sph_state *s, cudaStream_t st) {
  int64_t n = s->n;
  if (n == 0) return;
  { k_pack<<<nblk(n, 256), 256, 0, st>>>(s->x[0], s->x[1], s->x[2], s->v[0], s->v[1], s->v[2], s->h, s->m, s->rho, n,
                                       s->dim, s->inst_off, s->ninst, c->tree.inst_lo, c->units, c->pk); ++sph::g_launches; }
}

void tree_build(sph_ctx *c, const sph_state *s, int leaf_size, int max_depth, cudaStream_t st, bool pack) {
  Tree &T = c->tree;
  const int64_t n = s->n;
  const int ninst = s->ninst > 0 ? s->ninst : 1;
  const int dim = s->dim;
  T.leaf_size = leaf_size;
  T.max_depth = max_depth;
  T.packed_walk = (c->tune.plain_forms == 0 && T.cap_nodes <= kPackedSkip && max_depth <= 31) ? 1 : 0;
  T.perm_identity = 0;
  T.dim = dim;
  T.ninst = ninst;
  T.n = n;
  int ibits = 0;
  while ((1 << ibits) < ninst) ++ibits;
  const int bits = dim * max_depth + ibits, passes = sort_passes(bits);
  const bool wide = n >= 65536;  // see k_node_scan
  const int node_tiles = nblk(n + 1, wide ? 1024 : 256), group_tiles = nblk(T.cap_nodes, 256);
  uint32_t *node_state = T.look + kLookFixed + (int64_t)passes * nblk(n, kSortTile) * 256;
  uint32_t *group_state = node_state + node_tiles;
  const int64_t words = group_state + group_tiles - T.look;
  { k_tree_init<<<std::min(nblk(std::max<int64_t>(words, ninst), 256), 4 * c->num_sms), 256, 0, st>>>(T, words, ninst); ++sph::g_launches; }
  {
    BboxArgs A;
    memset(&A, 0, sizeof(A));
    for (int k = 0; k < 3; ++k) {
      A.x[k] = s->x[k];
      A.v[k] = s->v[k];
    }
    A.h = s->h;
    A.m = s->m;
    A.rho = s->rho;
    A.n = n;
    A.dim = dim;
    A.ninst = ninst;
    A.inst_off = s->inst_off;
    A.vscale = c->vscale;
    A.mt = c->mt;
    A.U = c->units;
    A.err = c->d_err;
    const int cols = (int)std::max<int64_t>(1, std::min<int64_t>(nblk(n / ninst + 1, 512), 8 * c->num_sms));
    { k_bbox<<<dim3(ninst, cols + 1), 256, 0, st>>>(A, T); ++sph::g_launches; }
  }
  if (n > 0) {
    { k_keys<<<std::min(nblk(n, 256), 8 * c->num_sms), 256, 0, st>>>(
          s->x[0], s->x[1], s->x[2], s->v[0], s->v[1], s->v[2], s->h, s->m, s->rho, n, dim, max_depth, s->inst_off,
          ninst, n <= kSmallSort ? 0 : passes, pack, c->pk, c->units, T); ++sph::g_launches; }
    sort_run(c, n, bits, st);
  } else {
    T.skey = T.keys[0];
    T.perm = T.vals[0];
  }
  KeyLevels K{T.skey, dim, max_depth};
  if (wide) k_node_scan<4><<<node_tiles, 256, 0, st>>>(K, n, leaf_size, s->inst_off, ninst, T, node_state, c->d_err);
  else k_node_scan<1><<<node_tiles, 256, 0, st>>>(K, n, leaf_size, s->inst_off, ninst, T, node_state, c->d_err);
  ++sph::g_launches;
  { k_node_emit<<<nblk(std::max<int64_t>(n, 1), 256), 256, 0, st>>>(K, n, leaf_size, s->inst_off, ninst, T.nstart, T); ++sph::g_launches; }
  const int mblocks = nblk(std::max<int64_t>(n, 1), 16);  // a leaf holds at least one particle
  if (dim == 3) k_moments<3><<<mblocks, 128, 0, st>>>(T, s->x[0], s->x[1], s->x[2], s->m, s->h);
  else k_moments<2><<<mblocks, 128, 0, st>>>(T, s->x[0], s->x[1], s->x[2], s->m, s->h);
  ++sph::g_launches;
  { k_node_finish<<<nblk(T.cap_nodes, 256), 256, 0, st>>>(T, dim, leaf_size, s->inst_off, ninst, c->units,
                                                        c->tune.walk_leaf); ++sph::g_launches; }
  { k_groups<<<std::min(group_tiles, 4 * c->num_sms), 256, 0, st>>>(T, s->inst_off, ninst, group_state, c->d_err); ++sph::g_launches; }
}

// ---------------------------------------------------------------------------
// In-place reorder of the caller's state along the tree
// ---------------------------------------------------------------------------
// All fields at once, doubles then ints: dst_f[i] = src_f[perm[i]].
constexpr int kMaxFields = 20;
struct FieldSet {
  const double *dsrc[kMaxFields];
  double *ddst[kMaxFields];
  const int32_t *isrc[2];
  int32_t *idst[2];
  int nd, ni;
};

__global__ void k_gather_fields(FieldSet F, const int32_t *__restrict__ perm, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t j = perm[i];
#pragma unroll 4
  for (int f = 0; f < F.nd; ++f) F.ddst[f][i] = F.dsrc[f][j];
  for (int f = 0; f < F.ni; ++f) F.idst[f][i] = F.isrc[f][j];
}

// Back into the state's arrays, perm[i] = i, and the FP32 views of the state
// in its new order
__global__ void k_copy_back(FieldSet F, int32_t *__restrict__ perm, int64_t n, int dim, const sph_state s,
                            const double *__restrict__ ilo, const Units *__restrict__ U, PackedF32 pk) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
#pragma unroll 4
  for (int f = 0; f < F.nd; ++f) F.ddst[f][i] = F.dsrc[f][i];
  for (int f = 0; f < F.ni; ++f) F.idst[f][i] = F.isrc[f][i];
  perm[i] = (int32_t)i;
  const int inst = inst_of(s.inst_off, s.ninst, i);
  pack_particle(pk, i, dim, s.x[0][i], s.x[1][i], dim == 3 ? s.x[2][i] : 0.0, s.v[0][i], s.v[1][i],
                dim == 3 ? s.v[2][i] : 0.0, s.h[i], s.m[i], s.rho[i], ilo + 3 * inst, U);
}

void tree_reorder_state(sph_ctx *c, sph_state *s, cudaStream_t st) {
  const int64_t n = s->n;
  if (n == 0) return;
  // scratch: the predicted-state and derivative buffers, free at this point
  StepBufs &B = c->st;
  double *scratch[kMaxFields] = {B.x[0], B.x[1], B.x[2], B.v[0], B.v[1], B.v[2], B.rho, B.u, B.dmg,
                                 B.d_x[0][0], B.d_x[0][1], B.d_x[0][2], B.d_v[0][0], B.d_v[0][1],
                                 B.d_v[0][2], B.d_rho[0], B.d_u[0], B.d_dmg[0], B.d_cs[0], B.gather};
  FieldSet G, R;
  memset(&G, 0, sizeof(G));
  auto add = [&](double *f) {
    if (!f) return;
    G.dsrc[G.nd] = f;
    G.ddst[G.nd] = scratch[G.nd];
    ++G.nd;
  };
  for (int ax = 0; ax < s->dim; ++ax) {
    add(s->x[ax]);
    add(s->v[ax]);
  }
  add(s->rho);
  add(s->u);
  add(s->m);
  add(s->h);
  add(s->dmg);
  if (s->S)
    for (int k = 0; k < nsym(s->dim); ++k) add(s->S + (int64_t)k * n);
  int32_t *iscr[2] = {B.gather_i, B.d_nact[0]};
  if (s->mat) {
    G.isrc[G.ni] = s->mat;
    G.idst[G.ni] = iscr[G.ni];
    ++G.ni;
  }
  if (s->id) {
    G.isrc[G.ni] = s->id;
    G.idst[G.ni] = iscr[G.ni];
    ++G.ni;
  }
  R = G;
  for (int f = 0; f < G.nd; ++f) {
    R.dsrc[f] = G.ddst[f];
    R.ddst[f] = const_cast<double *>(G.dsrc[f]);
  }
  for (int f = 0; f < G.ni; ++f) {
    R.isrc[f] = G.idst[f];
    R.idst[f] = const_cast<int32_t *>(G.isrc[f]);
  }
  { k_gather_fields<<<nblk(n, 256), 256, 0, st>>>(G, c->tree.perm, n); ++sph::g_launches; }
  { k_copy_back<<<nblk(n, 256), 256, 0, st>>>(R, c->tree.perm, n, s->dim, *s, c->tree.inst_lo, c->units, c->pk); ++sph::g_launches; }
  c->tree.perm_identity = 1;
}

// ---------------------------------------------------------------------------
// Node export (tests)
// ---------------------------------------------------------------------------
__global__ void k_export_nodes(Tree T, int64_t cap, int dim, int32_t *level, int64_t *cell, int64_t *count,
                               double *mass, double *com) {
  int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int nn = *T.nnodes;
  if (id >= nn || id >= cap) return;
  int l = T.level[id];
  unsigned long long pre = T.cell[id] & ((l * dim >= 64) ? ~0ULL : ((1ULL << (l * dim)) - 1ULL));
  level[id] = l;
  count[id] = T.end[id] - T.first[id];
  mass[id] = T.mass[id];
  if (dim == 3) {
    cell[3 * id] = (int64_t)compact3(pre);
    cell[3 * id + 1] = (int64_t)compact3(pre >> 1);
    cell[3 * id + 2] = (int64_t)compact3(pre >> 2);
  } else {
    cell[3 * id] = (int64_t)compact2(pre);
    cell[3 * id + 1] = (int64_t)compact2(pre >> 1);
    cell[3 * id + 2] = 0;
  }
  for (int ax = 0; ax < 3; ++ax) com[3 * id + ax] = T.com[ax * T.cap_nodes + id];
}

void export_nodes(sph_ctx *c, int64_t cap, int32_t *level, int64_t *cell, int64_t *count, double *mass, double *com,
                  cudaStream_t st) {
  { k_export_nodes<<<nblk(cap, 256), 256, 0, st>>>(c->tree, cap, c->tree.dim, level, cell, count, mass, com); ++sph::g_launches; }
}

}  // namespace sph
