// Tree construction on the device: root geometry, leaf binning, a stable LSD
// radix sort of (leaf key, original index), leaf ranges, the gather of
// positions/weights into leaf order, and the adaptive octree.
//
// Leaf boxes are numbered lexicographically, x fastest.  A point's leaf
// coordinate is floor((x - lo) / s_L) with s_L = size / 2^L, evaluated with
// round-to-nearest operations only, so the binning is reproducible.
//
// What bounds it: on small inputs the chain of launches (a binning, three scan
// and five sorting launches per 8 key bits came to 25 of a 6,000-point call's 28
// and to 100 of its 240 us), on large ones memory and the FP64 pipe (two lanes a
// cycle).  So a set of at most kSmallSort points is binned, sorted, gathered and
// ranged by one block in shared memory; a larger one takes one binning launch
// (keys and all digits' histograms), one launch per 8 key bits (a block ranks
// its tile, finds the digits' offsets by decoupled look-back over the earlier
// tiles and writes runs), the last of which also gathers; and the points are
// read as they come (double or float) and handled as pairs of floats.
#include <algorithm>

#include "adaptive.cuh"
#include "dwf.cuh"
#include "fmm_internal.cuh"

namespace {

__device__ void set_leaf_side(Geom* g, int L) {
  g->s_leaf = __ddiv_rn(g->size, (double)(1 << L));
  g->inv_s_leaf = 1.0 / g->s_leaf;
  g->m2l_count = 0;
  g->p2p_pairs = 0;
}

// (one block; also clears the sort's histograms and tickets, if any)
__global__ void k_geom_fixed(Geom* g, double lo0, double lo1, double lo2, double size, int L,
                             int* clear, int nclear) {
  for (int i = threadIdx.x; i < nclear; i += blockDim.x) clear[i] = 0;
  if (threadIdx.x != 0) return;
  g->lo[0] = lo0;
  g->lo[1] = lo1;
  g->lo[2] = lo2;
  g->size = size;
  g->flag = 0;
  set_leaf_side(g, L);
}

// per-block min/max over the sources and targets (bounding cube of the root)
template <int D, typename TI>
__global__ void k_bbox_partial(int64_t ns, const TI* __restrict__ src, int64_t nt,
                               const TI* __restrict__ tgt, double* out) {
  __shared__ double smin[D][256], smax[D][256];
  double mn[D], mx[D];
  for (int k = 0; k < D; ++k) {
    mn[k] = INFINITY;
    mx[k] = -INFINITY;
  }
  const int64_t n = ns + nt;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const TI* x = i < ns ? src + i * D : tgt + (i - ns) * D;
    for (int k = 0; k < D; ++k) {
      mn[k] = fmin(mn[k], (double)x[k]);
      mx[k] = fmax(mx[k], (double)x[k]);
    }
  }
  for (int k = 0; k < D; ++k) {
    smin[k][threadIdx.x] = mn[k];
    smax[k][threadIdx.x] = mx[k];
  }
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s)
      for (int k = 0; k < D; ++k) {
        smin[k][threadIdx.x] = fmin(smin[k][threadIdx.x], smin[k][threadIdx.x + s]);
        smax[k][threadIdx.x] = fmax(smax[k][threadIdx.x], smax[k][threadIdx.x + s]);
      }
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int k = 0; k < D; ++k) {
      out[(blockIdx.x * 2 + 0) * 3 + k] = smin[k][0];
      out[(blockIdx.x * 2 + 1) * 3 + k] = smax[k][0];
    }
}

// root = cube with corner at the minimum and side = the largest extent
template <int D>
__global__ void k_bbox_final(int nblk, const double* part, Geom* g, int L, int* clear,
                             int nclear) {
  for (int i = threadIdx.x; i < nclear; i += blockDim.x) clear[i] = 0;
  if (threadIdx.x != 0) return;
  double mn[3] = {0, 0, 0}, mx[3] = {0, 0, 0};
  for (int k = 0; k < D; ++k) {
    mn[k] = INFINITY;
    mx[k] = -INFINITY;
  }
  for (int b = 0; b < nblk; ++b)
    for (int k = 0; k < D; ++k) {
      mn[k] = fmin(mn[k], part[(b * 2 + 0) * 3 + k]);
      mx[k] = fmax(mx[k], part[(b * 2 + 1) * 3 + k]);
    }
  double size = 0.0;
  for (int k = 0; k < D; ++k) size = fmax(size, mx[k] - mn[k]);
  if (!(size > 0.0) || !isfinite(size)) size = 1.0;
  for (int k = 0; k < 3; ++k) g->lo[k] = (k < D && isfinite(mn[k])) ? mn[k] : 0.0;
  g->size = size;
  g->flag = 0;
  set_leaf_side(g, L);
}

}  // namespace

// (x - lo) / s rounded as an IEEE division.  The product with 1/s differs
// from the quotient by at most an ulp, which matters only when the quotient is
// within an ulp of an integer (a box face); those rare points take the exact
// division, so every point lands in the same leaf as with the division.
__device__ __forceinline__ double leaf_coord(double x, double lo, double s, double inv_s) {
  const double d = __dsub_rn(x, lo);
  const double t = d * inv_s;
  if (fabs(t - rint(t)) < 1e-6) return __ddiv_rn(d, s);
  return t;
}

namespace {

// exclusive scan of one value per thread over the block (at most 1024 threads)
__device__ int block_exclusive_scan(int v, int* smem, int* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int x = v;
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) smem[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int nw = blockDim.x >> 5;
    int s = lane < nw ? smem[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    smem[lane] = s;
  }
  __syncthreads();
  int incl = x + (wid > 0 ? smem[wid - 1] : 0);
  if (total) *total = smem[(blockDim.x >> 5) - 1];
  __syncthreads();
  return incl - v;
}

// ---- coordinates as pairs of floats -----------------------------------------
// x = h + l to about 48 bits (dw_bits: no FP64 instruction); false for what the
// float exponents cannot hold
struct FPair {
  float h, l;
};
__device__ __forceinline__ bool to_pair(double x, FPair* o) { return dw_bits(x, &o->h, &o->l); }
__device__ __forceinline__ bool to_pair(float x, FPair* o) {
  o->h = x;
  o->l = 0.f;
  return fabsf(x) < 1e35f;  // (false for NaN)
}

// the leaf grid along one axis: lo, the leaf side s and 1/s as pairs
struct AxisGrid {
  FPair lo, s, inv;
  bool ok;
};
struct LeafGrid {
  AxisGrid a[3];
};
__device__ __forceinline__ void load_grid(const Geom* g, int D, LeafGrid* out) {
  if (threadIdx.x < 3) {
    AxisGrid a;
    a.ok = to_pair(threadIdx.x < D ? g->lo[threadIdx.x] : 0.0, &a.lo);
    a.ok = to_pair(g->s_leaf, &a.s) && a.ok;
    a.ok = to_pair(g->inv_s_leaf, &a.inv) && a.ok;
    out->a[threadIdx.x] = a;
  }
}

// leaf coordinate of x along axis k: a float estimate, off by far less than
// 1e-3 leaf sides (t <= 1024: 3 roundings of 2^-24, and the pairs' 2^-46 of
// |x|, |lo|); points that close to a face take the FP64 path (identical to the
// division) for the exact leaf.  *bad: outside the root, clamped.
template <typename TI>
__device__ __forceinline__ int leaf_of(TI xv, const AxisGrid& a, const Geom* g, int k, int nl,
                                       bool* bad) {
  FPair p;
  if (to_pair(xv, &p) && a.ok && (fabsf(p.h) + fabsf(a.lo.h)) * a.inv.h < 1e9f) {
    const float t = ((p.h - a.lo.h) + (p.l - a.lo.l)) * a.inv.h;
    if (t >= 0.001f && t <= (float)nl - 0.001f && fabsf(t - rintf(t)) > 0.001f)
      return min((int)t, nl - 1);
  }
  const double t = leaf_coord((double)xv, g->lo[k], g->s_leaf, g->inv_s_leaf);
  if (!(t >= 0.0) || t > (double)nl) *bad = true;
  return (t >= 0.0) ? (int)fmin(floor(t), (double)(nl - 1)) : 0;  // NaN -> 0
}

// sort key of a point: its leaf, lexicographic (x fastest), or the Morton code
// of its box at the deepest level of an adaptive tree
template <int D, typename TI, bool MORTON>
__device__ __forceinline__ uint32_t key_of(const TI* __restrict__ x, const LeafGrid& lg,
                                           const Geom* g, int L, bool* bad) {
  const int nl = 1 << L;
  int c[3] = {0, 0, 0};
#pragma unroll
  for (int k = 0; k < D; ++k) c[k] = leaf_of<TI>(x[k], lg.a[k], g, k, nl, bad);
  if (MORTON) return morton3(c[0], c[1], c[2], L);
  uint32_t key = 0;
#pragma unroll
  for (int k = D - 1; k >= 0; --k) key = key * (uint32_t)nl + (uint32_t)c[k];
  return key;
}

// ---- the gather ----------------------------------------------------------------
// What a sorted point is written as: FP64 SoA copies, the float path's
// (x - c_own)/s and weight (c_own the centre of its leaf), or an adaptive
// tree's FP64 SoA copies with, for the sources of the float modes, x split into
// two floats, hi = fl(x) (and the weight) and lo = fl(x - hi).
enum GatherMode { kGatherSoa, kGatherRel, kGatherAdapt };
struct SortOut {
  double* o[3];
  double* w;
  int* perm;
  float4* rel;
  float4* hi;
  float4* lo;
};

__device__ __forceinline__ void two_sum(float a, float b, float* s, float* e) {
  *s = __fadd_rn(a, b);
  const float bb = __fadd_rn(*s, -a);
  *e = __fadd_rn(__fadd_rn(a, -__fadd_rn(*s, -bb)), __fadd_rn(b, -bb));
}

// (x - c)/s for the leaf b along an axis, c = lo + (b + 1/2) s, in float pairs;
// the FP64 form spent 5 FP64 instructions a coordinate (a float2double-bound
// 124 us of a 4M-point gather).  The pairs are off by about 2^-48 of (|x| + |lo|)/s, the
// result's rounding by 2^-26 at most, so they serve roots near the origin: against
// exact arithmetic the FP64 form and this one are off by 1.490e-8 and 1.495e-8
// at most (rms 6.51e-9 both) at (|x| + |lo|)/s = 2^14.4, by 1.49e-8 and 1.8e-8 at
// 2^20.5 and by 1.49e-8 and 1.9e-7 at 2^25.  Further out: FP64.
constexpr float kPairReach = 16384.f;
template <typename TI>
__device__ __forceinline__ float rel_coord(TI xv, const AxisGrid& a, const Geom* g, int k,
                                           uint32_t b) {
  FPair p;
  if (to_pair(xv, &p) && a.ok && (fabsf(p.h) + fabsf(a.lo.h)) * a.inv.h <= kPairReach) {
    const float bh = (float)b + 0.5f;
    const float q = __fmul_rn(bh, a.s.h);
    const float ql = __fmaf_rn(bh, a.s.l, __fmaf_rn(bh, a.s.h, -q));
    float ch, ce, dh, de;
    two_sum(a.lo.h, q, &ch, &ce);
    const float cl = __fadd_rn(ce, __fadd_rn(a.lo.l, ql));
    two_sum(p.h, -ch, &dh, &de);
    const float dl = __fadd_rn(de, __fadd_rn(p.l, -cl));
    return __fmaf_rn(dh, a.inv.h, __fmaf_rn(dh, a.inv.l, __fmul_rn(dl, a.inv.h)));
  }
  const double t = ((double)xv - g->lo[k]) * g->inv_s_leaf;
  return (float)(t - ((double)b + 0.5));
}

template <int D, typename TI, GatherMode M>
__device__ __forceinline__ void gather_point(const SortOut& o, int i, uint32_t key, int j,
                                             const TI* __restrict__ x, const TI* __restrict__ w,
                                             const LeafGrid& lg, const Geom* g, int L) {
  o.perm[i] = j;
  TI v[3] = {0, 0, 0};
#pragma unroll
  for (int k = 0; k < D; ++k) v[k] = x[(int64_t)j * D + k];
  const TI wj = w ? w[j] : (TI)0;
  if (M == kGatherRel) {
    const uint32_t m = (1u << L) - 1u;
    float u[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) u[k] = rel_coord<TI>(v[k], lg.a[k], g, k, (key >> (L * k)) & m);
    o.rel[i] = make_float4(u[0], u[1], u[2], (float)wj);
    return;
  }
#pragma unroll
  for (int k = 0; k < D; ++k) o.o[k][i] = (double)v[k];
  if (w) o.w[i] = (double)wj;
  if (M == kGatherAdapt && o.hi) {
    float h[3], l[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      h[k] = (float)v[k];
      l[k] = sizeof(TI) == 4 ? 0.f : (float)((double)v[k] - (double)h[k]);
    }
    o.hi[i] = make_float4(h[0], h[1], h[2], (float)wj);
    o.lo[i] = make_float4(l[0], l[1], l[2], 0.f);
  }
}

// first position of the sorted keys [0, n) that is >= v
template <typename PTR>
__device__ __forceinline__ int key_lower_bound(PTR a, int n, uint32_t v) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a[mid] < v) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// ---- small sets: one block, in shared memory -------------------------------------
constexpr int kSmallSort = 8192;
constexpr int kSmallThreads = 1024;
constexpr int kSmallRounds = kSmallSort / kSmallThreads;  // 32-point rounds per warp
constexpr int kSmallStarts = 8 * kSmallSort;  // leaf ranges found by the same block up to this
constexpr size_t kSmallSmem = 2 * kSmallSort * (sizeof(uint32_t) + sizeof(uint16_t)) +
                              32 * 256 * sizeof(int);
template <typename TI>
struct SmallJob {
  int n;
  const TI* x;
  const TI* w;
  SortOut out;
  uint32_t* keys;  // sorted keys, or null
  int* start;      // leaf ranges, or null
};
template <typename TI>
struct SmallJobs {
  SmallJob<TI> job[2];
};

// one block per set: bin, LSD radix sort by 8 bits (a warp ranks a contiguous
// run of points, so equal keys keep their order), gather, leaf ranges
template <int D, typename TI, GatherMode M>
__global__ void __launch_bounds__(kSmallThreads)
    k_sort_small(const __grid_constant__ SmallJobs<TI> jobs, const Geom* __restrict__ g, int L,
                 int bits, int nleaf, int* flag) {
  const SmallJob<TI>& J = jobs.job[blockIdx.x];
  extern __shared__ __align__(16) unsigned char smraw[];
  uint32_t* ka = reinterpret_cast<uint32_t*>(smraw);
  uint32_t* kb = ka + kSmallSort;
  uint16_t* va = reinterpret_cast<uint16_t*>(kb + kSmallSort);
  uint16_t* vb = va + kSmallSort;
  int(*cnt)[256] = reinterpret_cast<int(*)[256]>(vb + kSmallSort);  // [32 warps]
  __shared__ LeafGrid lg;
  __shared__ int sm[32];
  const int n = J.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  load_grid(g, D, &lg);
  __syncthreads();
  bool bad = false;
  for (int i = threadIdx.x; i < n; i += kSmallThreads) {
    ka[i] = key_of<D, TI, M == kGatherAdapt>(J.x + (int64_t)i * D, lg, g, L, &bad);
    va[i] = (uint16_t)i;
  }
  if (bad) atomicOr(flag, 1);
  // rounds of 32 points per warp, no more than the set needs
  const int rounds = (n + kSmallThreads - 1) / kSmallThreads;
  const int base = warp * rounds * 32;
  for (int shift = 0; shift < bits; shift += 8) {
    __syncwarp();
    for (int b = lane; b < 256; b += 32) cnt[warp][b] = 0;
    __syncthreads();  // the keys (and the previous pass' writes) are in place
    int rank[kSmallRounds];
#pragma unroll
    for (int r = 0; r < kSmallRounds; ++r) {
      if (r >= rounds) break;
      const int i = base + 32 * r + lane;
      const unsigned dig = i < n ? (ka[i] >> shift) & 255u : 256u;
      const unsigned peers = __match_any_sync(0xffffffffu, dig);
      const int before = __popc(peers & ((1u << lane) - 1u));
      const int have = dig < 256u ? cnt[warp][dig] : 0;
      rank[r] = have + before;
      __syncwarp();
      if (dig < 256u && before == 0) cnt[warp][dig] = have + __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    int tot = 0;
    if (threadIdx.x < 256)
      for (int w = 0; w < 32; ++w) {
        const int c = cnt[w][threadIdx.x];
        cnt[w][threadIdx.x] = tot;
        tot += c;
      }
    const int at = block_exclusive_scan(threadIdx.x < 256 ? tot : 0, sm, nullptr);
    if (threadIdx.x < 256)
      for (int w = 0; w < 32; ++w) cnt[w][threadIdx.x] += at;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSmallRounds; ++r) {
      if (r >= rounds) break;
      const int i = base + 32 * r + lane;
      if (i < n) {
        const uint32_t key = ka[i];
        const int pos = cnt[warp][(key >> shift) & 255u] + rank[r];
        kb[pos] = key;
        vb[pos] = va[i];
      }
    }
    uint32_t* kt = ka;
    ka = kb;
    kb = kt;
    uint16_t* vt = va;
    va = vb;
    vb = vt;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += kSmallThreads) {
    gather_point<D, TI, M>(J.out, i, ka[i], va[i], J.x, J.w, lg, g, L);
    if (J.keys) J.keys[i] = ka[i];
  }
  if (J.start)
    for (int b = threadIdx.x; b <= nleaf; b += kSmallThreads)
      J.start[b] = key_lower_bound(ka, n, (uint32_t)b);
}

// leaf ranges: start[b] = first sorted point of a leaf >= b (b = 0 .. nleaf)
__global__ void k_starts(int n, const uint32_t* __restrict__ keys, int nleaf,
                         int* __restrict__ start) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b <= nleaf) start[b] = key_lower_bound(keys, n, (uint32_t)b);
}

// ---- large sets -------------------------------------------------------------------
constexpr int kMaxPass = 4;                      // 8 key bits each
constexpr int kTileThreads = 256, kTileItems = 16;
constexpr int kTile = kTileThreads * kTileItems;
// scratch at the head of vals_a, per point set: the digits' histograms and a
// ticket per pass; after both sets', the look-back words of the set being sorted
constexpr int kSortHead = kMaxPass * 256 + 8;

// keys and the histograms of all their digits; clears the look-back words
template <int D, typename TI, bool MORTON>
__global__ void __launch_bounds__(256)
    k_bin(int n, const TI* __restrict__ x, const Geom* __restrict__ g, int L, int npass,
          uint32_t* __restrict__ keys, int* __restrict__ hist, uint32_t* __restrict__ look,
          int nlook, int* flag) {
  __shared__ LeafGrid lg;
  __shared__ int h[kMaxPass][256];
  for (int p = 0; p < kMaxPass; ++p) h[p][threadIdx.x] = 0;
  load_grid(g, D, &lg);
  __syncthreads();
  const int step = gridDim.x * blockDim.x, first = blockIdx.x * blockDim.x + threadIdx.x;
  for (int i = first; i < nlook; i += step) look[i] = 0;
  bool bad = false;
  for (int i = first; i < n; i += step) {
    const uint32_t key = key_of<D, TI, MORTON>(x + (int64_t)i * D, lg, g, L, &bad);
    keys[i] = key;
    for (int p = 0; p < npass; ++p) atomicAdd(&h[p][(key >> (8 * p)) & 255u], 1);
  }
  if (bad) atomicOr(flag, 1);
  __syncthreads();
  for (int p = 0; p < npass; ++p)
    if (h[p][threadIdx.x]) atomicAdd(&hist[p * 256 + threadIdx.x], h[p][threadIdx.x]);
}

// Look-back words: state << 30 | count (counts are below 2^30); a tile publishes
// its own count (kOwn), then its inclusive prefix (kIncl).  Tiles are handed out
// by a ticket, so every earlier tile has started, and publishes within
// microseconds.  The wait is bounded all the same (~1 ms): a waiter that gives up
// (returns 0) counts that tile itself, from what earlier launches wrote, so
// the result does not depend on it and no index is ever made from a missing count.
constexpr uint32_t kOwn = 1u << 30, kIncl = 2u << 30, kCount = kOwn - 1u;
constexpr long long kLookCycles = 2000000;
__device__ __forceinline__ uint32_t look_wait(const uint32_t* word, long long limit) {
  uint32_t v = *(volatile const uint32_t*)word;
  if (v >> 30) return v;
  const long long t0 = clock64();
  for (;;) {
    v = *(volatile const uint32_t*)word;
    if (v >> 30) return v;
    if (clock64() - t0 > limit) return 0;
  }
}

// one LSD pass over 8 key bits: vin null = identity; LAST also gathers
template <int D, typename TI, GatherMode M, bool LAST>
__global__ void __launch_bounds__(kTileThreads)
    k_sort_pass(int n, const uint32_t* __restrict__ kin, const int* __restrict__ vin,
                uint32_t* __restrict__ kout, int* __restrict__ vout, int shift,
                const int* __restrict__ hist, int* ticket, uint32_t* look, const SortOut out,
                const TI* __restrict__ x, const TI* __restrict__ w, const Geom* __restrict__ g,
                int L, long long limit) {
  constexpr int kW = kTileThreads / 32;
  __shared__ int cnt[kW][256];
  __shared__ int gbase[256];
  __shared__ uint32_t skey[kTile];
  __shared__ int sval[kTile];
  __shared__ int sm[32];
  __shared__ int stile;
  __shared__ LeafGrid lg;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, d = threadIdx.x;
  if (threadIdx.x == 0) stile = atomicAdd(ticket, 1);
  for (int q = 0; q < kW; ++q) cnt[q][d] = 0;
  if (LAST) load_grid(g, D, &lg);
  __syncthreads();
  const int tile = stile, t0 = tile * kTile;
  const int tn = min(kTile, n - t0);
  uint32_t key[kTileItems];
  int rank[kTileItems];
  // a warp takes a contiguous run of the tile, 32 points a round (stable)
  const int base = warp * (kTile / kW) + lane;
#pragma unroll
  for (int r = 0; r < kTileItems; ++r)
    key[r] = base + 32 * r < tn ? kin[t0 + base + 32 * r] : 0xffffffffu;
#pragma unroll
  for (int r = 0; r < kTileItems; ++r) {
    const unsigned dig = base + 32 * r < tn ? (key[r] >> shift) & 255u : 256u;
    const unsigned peers = __match_any_sync(0xffffffffu, dig);
    const int before = __popc(peers & ((1u << lane) - 1u));
    const int have = dig < 256u ? cnt[warp][dig] : 0;
    rank[r] = have + before;
    __syncwarp();
    if (dig < 256u && before == 0) cnt[warp][dig] = have + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  int tot = 0;  // digit d: this tile's count, its warps' offsets
#pragma unroll
  for (int q = 0; q < kW; ++q) {
    const int c = cnt[q][d];
    cnt[q][d] = tot;
    tot += c;
  }
  uint32_t* mine = look + (size_t)tile * 256 + d;
  *(volatile uint32_t*)mine = (tile == 0 ? kIncl : kOwn) | (uint32_t)tot;
  const int loc = block_exclusive_scan(tot, sm, nullptr);
  const int glob = block_exclusive_scan(hist[d], sm, nullptr);
  if (tile > 0) {
    uint32_t before = 0;
    for (int t = tile - 1; t >= 0; --t) {
      uint32_t v = look_wait(look + (size_t)t * 256 + d, limit);
      if (v == 0) {  // gave up: the (full) tile's keys of digit d
        v = kOwn;
        for (int i = 0; i < kTile; ++i)
          v += ((kin[t * kTile + i] >> shift) & 255u) == (unsigned)d ? 1u : 0u;
      }
      before += v & kCount;
      if (v & kIncl) break;
    }
    *(volatile uint32_t*)mine = kIncl | (before + (uint32_t)tot);
    gbase[d] = glob + (int)before - loc;
  } else {
    gbase[d] = glob - loc;
  }
#pragma unroll
  for (int q = 0; q < kW; ++q) cnt[q][d] += loc;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kTileItems; ++r) {
    const int i = base + 32 * r;
    if (i < tn) {
      const int pos = cnt[warp][(key[r] >> shift) & 255u] + rank[r];
      skey[pos] = key[r];
      sval[pos] = vin ? vin[t0 + i] : t0 + i;
    }
  }
  __syncthreads();
#pragma unroll 4
  for (int i = threadIdx.x; i < tn; i += kTileThreads) {
    const uint32_t k = skey[i];
    const int pos = gbase[(k >> shift) & 255u] + i;
    kout[pos] = k;
    if (LAST) gather_point<D, TI, M>(out, pos, k, sval[i], x, w, lg, g, L);
    else vout[pos] = sval[i];
  }
}

// ---- adaptive octree (adaptive.cuh) ----------------------------------------
// the root box, the level offsets, and the level kernels' tickets and look-back words
__global__ void k_atree_root(int* lev, int* par, uint32_t* key, int* s0, int* s1, int* t0,
                             int* t1, int ns, int nt, int* dlo, int nlo, int* ticket, int nticket,
                             uint32_t* look, int nlook, int* bnd, int nbnd) {
  const int i0 = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  for (int i = i0; i < nlook; i += step) look[i] = 0;
  for (int i = i0; i < nticket; i += step) ticket[i] = 0;
  for (int i = i0; i < nbnd; i += step) bnd[i] = (i % 6) < 3 ? 0x7fffffff : -1;
  for (int l = i0; l < nlo; l += step) dlo[l] = l == 0 ? 0 : 1;  // the root alone
  if (i0 != 0) return;
  dlo[nlo] = 0;  // overflow flag
  lev[0] = 0;
  par[0] = -1;
  key[0] = 0;
  s0[0] = 0;
  s1[0] = ns;
  t0[0] = 0;
  t1[0] = nt;
}

// per-level coordinate bounds of the boxes of levels >= 2 (the windows of the
// adaptive tensor-core M2L): bnd[6 l + k] = min, bnd[6 l + 3 + k] = max
__global__ void k_abounds(const int* __restrict__ dlo, int D, const int* __restrict__ lev,
                          const uint32_t* __restrict__ key, int* __restrict__ bnd) {
  // boxes are stored level by level, so a warp mostly holds one level: reduce
  // over the lanes of each level first, one atomic per level and warp
  const int b = blockIdx.x * blockDim.x + threadIdx.x;  // the grid covers whole warps
  int l = -1, c[3] = {0, 0, 0};
  if (b < dlo[D + 1] && lev[b] >= 2) {
    l = lev[b];
    demorton3(key[b], l, c);
  }
  const unsigned grp = __match_any_sync(0xffffffffu, l);
  if (l < 0) return;
  const bool lead = (threadIdx.x & 31) == __ffs(grp) - 1;
  for (int k = 0; k < 3; ++k) {
    const int mn = __reduce_min_sync(grp, c[k]), mx = __reduce_max_sync(grp, c[k]);
    if (lead) {
      atomicMin(&bnd[6 * l + k], mn);
      atomicMax(&bnd[6 * l + 3 + k], mx);
    }
  }
}

// dense index of the coarse levels: grid[(8^l - 1)/7 + code] = box
__global__ void k_agrid_fill(int nbox, int glev, const uint32_t* __restrict__ key,
                             const int* __restrict__ lev, int* __restrict__ grid) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nbox || lev[b] > glev) return;
  grid[agrid_offset(lev[b]) + key[b]] = b;
}

// first position in sorted[lo, hi) whose code is >= v
__device__ inline int lower_bound_u32(const uint32_t* a, int lo, int hi, uint32_t v) {
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a[mid] < v) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// A box's child ranges are the boundaries of its octants 1..7 in the sorted
// source and target codes: fourteen binary searches, one per lane of a group
// of 16 lanes (lanes 0..6 sources, 8..14 targets), so that a level's kernels
// wait for one search's chain of dependent loads, not fourteen.  Every lane of
// the group gets all boundaries sb[0..8], tb[0..8] by shuffles.
constexpr int kBoxLanes = 16;
__device__ __forceinline__ void child_bounds_group(const uint32_t* skey, const uint32_t* tkey,
                                                   bool live, uint32_t key, int l, int D, int s0,
                                                   int s1, int t0, int t1, int* sb, int* tb) {
  const int k = threadIdx.x & (kBoxLanes - 1);
  int v = 0;
  if (live && k != 7 && k != 15) {
    const int ci = (k & 7) + 1;
    const uint32_t c = ((key << 3) | (uint32_t)ci) << (3 * (D - l - 1));
    v = k < 8 ? lower_bound_u32(skey, s0, s1, c) : lower_bound_u32(tkey, t0, t1, c);
  }
  sb[0] = s0;
  tb[0] = t0;
#pragma unroll
  for (int ci = 1; ci < 8; ++ci) {
    sb[ci] = __shfl_sync(0xffffffffu, v, ci - 1, kBoxLanes);
    tb[ci] = __shfl_sync(0xffffffffu, v, ci + 7, kBoxLanes);
  }
  sb[8] = s1;
  tb[8] = t1;
}

constexpr int kLevelThreads = 256;
constexpr int kLevelBoxes = kLevelThreads / kBoxLanes;
static_assert(kLevelBoxes == kATileBoxes, "look-back words per level");

// children of the (full) tile of boxes from b on, counted by a warp, two boxes at a
// time.  Not inlined, and the launch bound of the kernel that calls it keeps
// eight blocks an SM: inlined it cost fifteen registers, three blocks and 86 of
// then 479 us on the levels of a 2M-point tree.
__device__ __noinline__ int tile_children(int b, int max_leaf, int l, int D, const uint32_t* key,
                                          const int* s0, const int* s1, const int* t0,
                                          const int* t1, const uint32_t* skey,
                                          const uint32_t* tkey) {
  int kids = 0;
  for (int i = 0; i < kLevelBoxes; i += 2) {
    const int e = b + i + (int)threadIdx.x / kBoxLanes;
    const bool split = (s1[e] - s0[e]) + (t1[e] - t0[e]) > max_leaf && l < D;
    int sb[9], tb[9];
    child_bounds_group(skey, tkey, split, key[e], l, D, s0[e], s1[e], t0[e], t1[e], sb, tb);
    if (split)
      for (int ci = 0; ci < 8; ++ci) kids += (sb[ci + 1] > sb[ci] || tb[ci + 1] > tb[ci]) ? 1 : 0;
  }
  return kids + __shfl_xor_sync(0xffffffffu, kids, kBoxLanes);
}

// One level of the tree in one launch: the split decision of every box of level
// l (boxes dlo[l] .. dlo[l+1]; level offsets kept on the device), its non-empty
// children appended behind the level in box order, and dlo[l+2].  16 lanes a
// box (lane c < 8 writes child c), 16 boxes a tile; tiles are handed out by a
// ticket and find where their children go by look-back over the earlier tiles'
// counts.  A split, a clear, three scan and an emit launch per level took 60
// launches and 0.25 ms of a 60k-point tree, and on large ones ran over the bound
// on the level's boxes.  Past the capacity: raise dlo[nlo], add nothing.
__global__ void __launch_bounds__(kLevelThreads, 8)
    k_atree_level(int* __restrict__ dlo, int nlo, int cap, int l, int D, int max_leaf,
                  uint32_t* __restrict__ key, int* __restrict__ lev, int* __restrict__ par,
                  int* __restrict__ s0, int* __restrict__ s1, int* __restrict__ t0,
                  int* __restrict__ t1, const uint32_t* __restrict__ skey,
                  const uint32_t* __restrict__ tkey, int* __restrict__ leaf,
                  int* __restrict__ child, int* ticket, uint32_t* look, int* min_leaf,
                  long long limit) {
  __shared__ int stile, sbase, scount[kLevelBoxes];
  const int b0 = dlo[l], b1 = dlo[l + 1];
  const int tiles = (b1 - b0 + kLevelBoxes - 1) / kLevelBoxes;
  uint32_t* words = look + (b0 / kLevelBoxes + l);  // this level's (no overlap with others')
  const int grp = threadIdx.x / kBoxLanes, k = threadIdx.x & (kBoxLanes - 1);
  if (tiles == 0) {  // a level past the last split: carry the offset down
    if (blockIdx.x == 0 && threadIdx.x == 0) dlo[l + 2] = b1;
    return;
  }
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) stile = atomicAdd(ticket, 1);
    __syncthreads();
    const int tile = stile;
    if (tile >= tiles) return;
    const int b = b0 + tile * kLevelBoxes + grp;
    const bool live = b < b1;
    int bs0 = 0, bs1 = 0, bt0 = 0, bt1 = 0;
    uint32_t bkey = 0;
    bool split = false;
    if (live) {
      bs0 = s0[b], bs1 = s1[b], bt0 = t0[b], bt1 = t1[b], bkey = key[b];
      split = (bs1 - bs0) + (bt1 - bt0) > max_leaf && l < D;
    }
    int sb[9], tb[9];  // every lane of the block reaches the shuffles
    child_bounds_group(skey, tkey, live && split, bkey, l, D, bs0, bs1, bt0, bt1, sb, tb);
    int n = 0, before = 0;  // children of the box, and those ahead of child k
    if (split)
#pragma unroll
      for (int ci = 0; ci < 8; ++ci) {
        const int has = (sb[ci + 1] > sb[ci] || tb[ci + 1] > tb[ci]) ? 1 : 0;
        n += has;
        before += ci < k ? has : 0;
      }
    if (k == 0) scount[grp] = n;
    if (__syncthreads_or(live && !split) && threadIdx.x == 0 && *(volatile int*)min_leaf > l)
      atomicMin(min_leaf, l);
    if (threadIdx.x < 32) {  // the tile's count, then the earlier tiles' by look-back
      int tot = threadIdx.x < kLevelBoxes ? scount[threadIdx.x] : 0;
      for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
      if (threadIdx.x == 0)
        *(volatile uint32_t*)&words[tile] = (tile == 0 ? kIncl : kOwn) | (uint32_t)tot;
      uint32_t base = 0;
      for (int t = tile - 1; t >= 0; t -= 32) {  // 32 earlier tiles at a time
        const int at = t - (int)threadIdx.x;
        uint32_t v = at >= 0 ? look_wait(&words[at], limit) : kIncl;
        // lanes that gave up: the warp counts their tiles' children
        for (unsigned gone = __ballot_sync(0xffffffffu, v == 0); gone; gone &= gone - 1) {
          const int q = __ffs(gone) - 1;
          const int kids = tile_children(b0 + (t - q) * kLevelBoxes, max_leaf, l, D, key, s0, s1,
                                         t0, t1, skey, tkey);
          if ((int)threadIdx.x == q) v = kOwn | (uint32_t)kids;
        }
        const unsigned incl = __ballot_sync(0xffffffffu, (v & kIncl) != 0);
        const int last = incl ? __ffs(incl) - 1 : 31;  // nearest inclusive prefix
        uint32_t c = (int)threadIdx.x <= last ? v & kCount : 0u;
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        base += c;
        if (incl) break;
      }
      if (threadIdx.x == 0) {
        *(volatile uint32_t*)&words[tile] = kIncl | (base + (uint32_t)tot);
        sbase = (int)base;
        if (tile == tiles - 1) {  // the level's total (read by the next level's launch)
          const bool over = (int64_t)b1 + base + tot > cap;
          dlo[l + 2] = over ? b1 : b1 + (int)base + tot;
          if (over) dlo[nlo] = 1;
        }
      }
    }
    __syncthreads();
    if (live) {
      int pos = b1 + sbase + before;
      for (int q = 0; q < grp; ++q) pos += scount[q];
      if (k == 0) leaf[b] = split ? 0 : 1;
      if (k < 8) {
        const bool has = split && (sb[k + 1] > sb[k] || tb[k + 1] > tb[k]) && pos < cap;
        child[8 * b + k] = has ? pos : -1;
        if (has) {
          key[pos] = (bkey << 3) | (uint32_t)k;
          lev[pos] = l + 1;
          par[pos] = b;
          s0[pos] = sb[k];
          s1[pos] = sb[k + 1];
          t0[pos] = tb[k];
          t1[pos] = tb[k + 1];
        }
      }
    }
  }
}

// cycles a look-back waits (fmm_set_wait_limit shortens it for tests)
long long look_limit(const fmm_plan_s* P) {
  return P->tc_wait_cycles > 0 ? std::min(P->tc_wait_cycles, kLookCycles) : kLookCycles;
}

unsigned nblocks(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

template <int D, typename TI, GatherMode M>
cudaError_t sort_small(const SmallJobs<TI>& jobs, int njobs, const Workspace& ws, int L, int nleaf,
                       cudaStream_t st, int* nl) {
  // (per call: the attribute belongs to the current device's context)
  cudaFuncSetAttribute(k_sort_small<D, TI, M>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)kSmallSmem);
  k_sort_small<D, TI, M><<<njobs, kSmallThreads, kSmallSmem, st>>>(jobs, ws.geom, L, D * L, nleaf,
                                                                   &ws.geom->flag);
  ++*nl;
  return cudaGetLastError();
}

// sort one set of more than kSmallSort points; set 0 or 1 (its histograms).
// keys: where the sorted keys go (null: a scratch array, returned in *sorted)
template <int D, typename TI, GatherMode M>
cudaError_t sort_large(const Workspace& ws, int set, int n, const TI* x, const TI* w,
                       const SortOut& out, int L, uint32_t* keys, const uint32_t** sorted,
                       long long limit, cudaStream_t st, int* nl) {
  const int bits = D * L, npass = (bits + 7) / 8, tiles = (n + kTile - 1) / kTile;
  int* head = ws.vals_a + set * kSortHead;
  int* ticket = head + kMaxPass * 256;
  uint32_t* look = reinterpret_cast<uint32_t*>(ws.vals_a + 2 * kSortHead);
  const unsigned blocks = std::min<unsigned>(nblocks(n, 256), 152 * 16);
  k_bin<D, TI, M == kGatherAdapt><<<blocks, 256, 0, st>>>(
      n, x, ws.geom, L, npass, ws.keys_a, head, look, npass * tiles * 256, &ws.geom->flag);
  ++*nl;
  uint32_t* kin = ws.keys_a;
  uint32_t* kout = ws.keys_b;
  const int* vin = nullptr;
  for (int p = 0; p < npass; ++p) {
    const bool last = p == npass - 1;
    // values alternate between the scratch array and perm so that the last
    // pass, which writes perm, reads the scratch array
    int* vout = ((npass - 2 - p) & 1) ? out.perm : ws.vals_b;
    if (last && keys) kout = keys;
    uint32_t* lk = look + (size_t)p * tiles * 256;
    if (last)
      k_sort_pass<D, TI, M, true><<<tiles, kTileThreads, 0, st>>>(
          n, kin, vin, kout, nullptr, 8 * p, head + 256 * p, ticket + p, lk, out, x, w, ws.geom, L,
          limit);
    else
      k_sort_pass<D, TI, M, false><<<tiles, kTileThreads, 0, st>>>(
          n, kin, vin, kout, vout, 8 * p, head + 256 * p, ticket + p, lk, out, x, w, ws.geom, L,
          limit);
    ++*nl;
    vin = vout;
    std::swap(kin, kout);
  }
  *sorted = kin;
  return cudaGetLastError();
}

// sort the sources (and the targets, unless they are the sources) into leaf
// order with their leaf ranges
template <int D, typename TI, GatherMode M>
cudaError_t sort_uniform(const fmm_plan_s* P, const Workspace& ws, int64_t n_src, const TI* src,
                         const TI* w, int64_t n_tgt, const TI* tgt, bool shared, cudaStream_t st,
                         int* nl) {
  const int L = P->desc.levels, nleaf = (int)nbox_at(D, L);
  const SortOut outs[2] = {{{ws.sx[0], ws.sx[1], ws.sx[2]}, ws.sw, ws.sperm, ws.sxr, nullptr, nullptr},
                           {{ws.tx[0], ws.tx[1], ws.tx[2]}, nullptr, ws.tperm, ws.txr, nullptr, nullptr}};
  const int64_t n[2] = {n_src, n_tgt};
  const TI* x[2] = {src, tgt};
  int* start[2] = {ws.sstart, ws.tstart};
  const bool few = nleaf <= kSmallStarts;
  SmallJobs<TI> jobs{};
  int njobs = 0;
  cudaError_t e;
  for (int k = 0; k < (shared ? 1 : 2); ++k)
    if (n[k] <= kSmallSort)
      jobs.job[njobs++] = {(int)n[k], x[k], k == 0 ? w : nullptr, outs[k],
                           few ? nullptr : (k == 0 ? ws.keys_a : ws.keys_b),
                           few ? start[k] : nullptr};
  if (njobs && (e = sort_small<D, TI, M>(jobs, njobs, ws, L, nleaf, st, nl)) != cudaSuccess)
    return e;
  for (int k = 0; k < (shared ? 1 : 2); ++k) {
    // (a small set's keys are used before the other, larger set's sort reuses the arrays)
    if (n[k] > kSmallSort || few) continue;
    k_starts<<<nblocks(nleaf + 1, 256), 256, 0, st>>>((int)n[k], k == 0 ? ws.keys_a : ws.keys_b,
                                                      nleaf, start[k]);
    ++*nl;
  }
  for (int k = 0; k < (shared ? 1 : 2); ++k) {
    if (n[k] <= kSmallSort) continue;
    const uint32_t* sorted = nullptr;
    if ((e = sort_large<D, TI, M>(ws, k, (int)n[k], x[k], k == 0 ? w : nullptr, outs[k], L,
                                  nullptr, &sorted, look_limit(P), st, nl)) != cudaSuccess)
      return e;
    k_starts<<<nblocks(nleaf + 1, 256), 256, 0, st>>>((int)n[k], sorted, nleaf, start[k]);
    ++*nl;
  }
  return cudaGetLastError();
}

}  // namespace

template <typename TI>
static cudaError_t set_geom(const fmm_plan_s* P, const Workspace& ws, int64_t n_src, const TI* src,
                            int64_t n_tgt, const TI* tgt, cudaStream_t st, int* nl) {
  const fmm_plan_desc& d = P->desc;
  const int depth = d.levels > 0 ? d.levels : -d.levels;  // adaptive: deepest level
  const int clear = std::max(n_src, n_tgt) > kSmallSort ? 2 * kSortHead : 0;
  if (d.root_size > 0.0) {
    k_geom_fixed<<<1, 256, 0, st>>>(ws.geom, d.root_lo[0], d.root_lo[1],
                                    d.d == 3 ? d.root_lo[2] : 0.0, d.root_size, depth, ws.vals_a,
                                    clear);
    ++*nl;
    return cudaGetLastError();
  }
  const int nb = ws.nbbox_blocks;
  if (P->pd.d == 3) {
    k_bbox_partial<3, TI><<<nb, 256, 0, st>>>(n_src, src, n_tgt, tgt, ws.bbox);
    k_bbox_final<3><<<1, 256, 0, st>>>(nb, ws.bbox, ws.geom, depth, ws.vals_a, clear);
  } else {
    k_bbox_partial<2, TI><<<nb, 256, 0, st>>>(n_src, src, n_tgt, tgt, ws.bbox);
    k_bbox_final<2><<<1, 256, 0, st>>>(nb, ws.bbox, ws.geom, depth, ws.vals_a, clear);
  }
  *nl += 2;
  return cudaGetLastError();
}

cudaError_t launch_set_geom(const fmm_plan_s* P, const Workspace& ws, const PointSets& pts,
                            cudaStream_t st, int* nl) {
  if (pts.f32)
    return set_geom(P, ws, pts.n_src, (const float*)pts.src, pts.n_tgt, (const float*)pts.tgt, st,
                    nl);
  return set_geom(P, ws, pts.n_src, (const double*)pts.src, pts.n_tgt, (const double*)pts.tgt, st,
                  nl);
}

cudaError_t launch_build_tree(const fmm_plan_s* P, const Workspace& ws, const PointSets& pts,
                              cudaStream_t st, int* nl) {
  const bool shared = ws.tstart == ws.sstart;  // targets are the sources: sorted once
#define SORT_GO(DD, TT, MM)                                                                     \
  return sort_uniform<DD, TT, MM>(P, ws, pts.n_src, (const TT*)pts.src, (const TT*)pts.w,       \
                                  pts.n_tgt, (const TT*)pts.tgt, shared, st, nl)
  if (P->pd.d == 3 && ws.sxr) {  // the FP32 path keeps only the box-relative float4 copies
    if (pts.f32) SORT_GO(3, float, kGatherRel);
    SORT_GO(3, double, kGatherRel);
  }
  if (P->pd.d == 3) {
    if (pts.f32) SORT_GO(3, float, kGatherSoa);
    SORT_GO(3, double, kGatherSoa);
  }
  if (pts.f32) SORT_GO(2, float, kGatherSoa);
  SORT_GO(2, double, kGatherSoa);
#undef SORT_GO
}

namespace {

// sort both point sets of an adaptive tree by Morton code at depth D
template <typename TI>
cudaError_t sort_adaptive(const Workspace& ws, int D, int64_t n_src, const TI* src, const TI* w,
                          int64_t n_tgt, const TI* tgt, bool shared, long long limit,
                          cudaStream_t st, int* nl) {
  const SortOut outs[2] = {
      {{ws.sx[0], ws.sx[1], ws.sx[2]}, ws.sw, ws.sperm, nullptr, ws.asxh, ws.asxl},
      {{ws.tx[0], ws.tx[1], ws.tx[2]}, nullptr, ws.tperm, nullptr, nullptr, nullptr}};
  const int64_t n[2] = {n_src, n_tgt};
  const TI* x[2] = {src, tgt};
  uint32_t* keys[2] = {ws.skey, ws.tkey};
  SmallJobs<TI> jobs{};
  int njobs = 0;
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < (shared ? 1 : 2); ++k)
    if (n[k] > 0 && n[k] <= kSmallSort)
      jobs.job[njobs++] = {(int)n[k], x[k], k == 0 ? w : nullptr, outs[k], keys[k], nullptr};
  if (njobs) e = sort_small<3, TI, kGatherAdapt>(jobs, njobs, ws, D, 0, st, nl);
  for (int k = 0; k < (shared ? 1 : 2) && e == cudaSuccess; ++k) {
    if (n[k] <= kSmallSort) continue;
    const uint32_t* sorted = nullptr;
    e = sort_large<3, TI, kGatherAdapt>(ws, k, (int)n[k], x[k], k == 0 ? w : nullptr, outs[k], D,
                                        keys[k], &sorted, limit, st, nl);
  }
  return e;
}

}  // namespace

cudaError_t launch_build_adaptive(const fmm_plan_s* P, const Workspace& ws, const PointSets& pts,
                                  cudaStream_t st, int* nl, ATree* t, int* overflow) {
  const int D = -P->desc.levels;
  const int64_t n_src = pts.n_src, n_tgt = pts.n_tgt;
  *overflow = 0;
  const bool shared = ws.tkey == ws.skey;  // the targets are the sources, sorted once
  cudaError_t e =
      pts.f32 ? sort_adaptive(ws, D, n_src, (const float*)pts.src, (const float*)pts.w, n_tgt,
                              (const float*)pts.tgt, shared, look_limit(P), st, nl)
              : sort_adaptive(ws, D, n_src, (const double*)pts.src, (const double*)pts.w, n_tgt,
                              (const double*)pts.tgt, shared, look_limit(P), st, nl);
  if (e != cudaSuccess) return e;
  // Level by level without the host: the level offsets live on the device
  // (dlo[0..D+2], overflow flag at dlo[D+3]) and every level's kernels read
  // their box range there.  One read at the end.  The host sizes each
  // level's launches by a bound on its box count: level l+1 holds at most 8
  // children of each split box of level l, there are at most n / (max_leaf + 1)
  // split boxes (their point sets are disjoint), and no box is empty.
  const int nlo = D + 3;
  int* dlo = ws.aloff;
  int* dbnd = dlo + nlo + 1;  // [0]: smallest leaf level; 6 l ..: bounds of level l >= 2
  const int nbnd = 6 * (D + 2);
  const int cap = (int)ws.anb_cap;
  const int64_t npts = n_src + (shared ? 0 : n_tgt);
  const int64_t splits_cap = (n_src + n_tgt) / ((int64_t)P->desc.max_leaf + 1);
  int* ticket = ws.ascan;  // one per level
  uint32_t* look = ws.alook;
  const int nlook = (int)atree_look_words(cap, D);
  if (nlook > ws.alook_n || D + 1 > ws.ascan_n) return cudaErrorInvalidValue;
  k_atree_root<<<std::min<unsigned>(nblocks(nlook, 256), 152), 256, 0, st>>>(
      ws.alev, ws.apar, ws.akey, ws.as0, ws.as1, ws.at0, ws.at1, (int)n_src, (int)n_tgt, dlo, nlo,
      ticket, D + 1, look, nlook, dbnd, nbnd);
  ++*nl;
  int64_t bound = 1;  // boxes of level l at most
  for (int l = 0; l <= D; ++l) {
    const int64_t nb = std::max<int64_t>(1, std::min<int64_t>(bound, cap));
    k_atree_level<<<std::min<unsigned>(nblocks(nb, kLevelBoxes), 152 * 8), kLevelThreads, 0, st>>>(
        dlo, nlo, cap, l, D, P->desc.max_leaf, ws.akey, ws.alev, ws.apar, ws.as0, ws.as1, ws.at0,
        ws.at1, ws.skey, ws.tkey, ws.aleaf, ws.achild, ticket + l, look, dbnd,
        look_limit(P));
    ++*nl;
    bound = std::min<int64_t>(8 * std::min<int64_t>(bound, splits_cap), std::max<int64_t>(npts, 1));
  }
  // the levels' coordinate bounds (for the adaptive M2L's windows), read in the same copy
  k_abounds<<<nblocks(cap, 256), 256, 0, st>>>(dlo, D, ws.alev, ws.akey, dbnd);
  ++*nl;
  static_assert(sizeof(P->abnd) >= sizeof(int) * 6 * (FMM_MAX_ADEPTH + 2), "level bounds");
  int hlo[FMM_MAX_ADEPTH + 4 + 6 * (FMM_MAX_ADEPTH + 2)];
  cudaMemcpyAsync(hlo, dlo, sizeof(int) * (nlo + 1 + nbnd), cudaMemcpyDeviceToHost, st);
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
  std::copy(hlo + nlo + 1, hlo + nlo + 1 + nbnd, const_cast<fmm_plan_s*>(P)->abnd);
  if (hlo[nlo]) {
    *overflow = 1;
    return cudaSuccess;
  }
  int loff[FMM_MAX_ADEPTH + 2];
  int maxlev = 0;
  for (int l = 0; l <= D + 1; ++l) loff[l] = hlo[l];
  for (int l = 1; l <= D; ++l)
    if (hlo[l + 1] > hlo[l]) maxlev = l;
  t->key = ws.akey;
  t->lev = ws.alev;
  t->par = ws.apar;
  t->child = ws.achild;
  t->s0 = ws.as0;
  t->s1 = ws.as1;
  t->t0 = ws.at0;
  t->t1 = ws.at1;
  t->leaf = ws.aleaf;
  for (int l = 0; l <= FMM_MAX_ADEPTH + 1; ++l) t->loff[l] = l <= maxlev + 1 ? loff[l] : loff[maxlev + 1];
  t->maxlev = maxlev;
  t->min_leaf = std::min(P->abnd[0], maxlev);  // (the bounds of levels 0 and 1 are not used)
  // dense index of levels 0..glev (one load per lookup there)
  const int glev = std::min(maxlev, FMM_AGRID_LEVELS);
  const int nbox = loff[maxlev + 1];
  cudaMemsetAsync(ws.agrid, 0xff, sizeof(int) * (size_t)agrid_offset(glev + 1), st);
  k_agrid_fill<<<nblocks(nbox, 256), 256, 0, st>>>(nbox, glev, ws.akey, ws.alev, ws.agrid);
  ++*nl;
  t->grid = ws.agrid;
  t->grid_levels = glev;
  return cudaGetLastError();
}
