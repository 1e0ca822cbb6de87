// Tensor-core M2L (tcgen05, kind::tf32 / kind::f16) -- eq. (m2l_toeplitz) grouped by
// translation offset into dense contractions on the fifth-generation tensor
// cores, with the accumulator in TMEM.
//
// For a level with half-grid size H = 2^(l-1), write every box as 2T + pi
// (T its parent's coordinate, pi in {0,1}^3 its position in the parent).
// A target of class pi receives, from source child sigma of the parent
// T + delta (delta in {-1,0,1}^3), the translation with offset
// h = pi - sigma - 2 delta, whenever h is not adjacent (max |h_k| >= 2).
// For a fixed (pi, sigma, delta) the sources of a tile of targets T are the
// same tile of parents shifted by delta, so with the multipoles stored
// parity-split, Bpar[sigma][Tz][Ty][Tx][q], one 5-D TMA box (zero-filled
// outside the domain) is a dense operand, and so is the offset matrix
//   A_h[i][q] = Ht_h[i + q]   (i, q in j).
//
// Orientation.  A pair of CTAs (cta_group::2, a cluster) works on one tile: the
// MMA's M dimension holds 256 target parents (128 TMEM lanes in each CTA), N
// holds the local coefficients i and K the multipole coefficients q:
//   D[T][i] += sum_q Bpar[sigma][T + delta][q] * A_h[i][q],
// so |j| is padded only to the pair's N granularity of 32 (130 -> 160 for the
// biharmonic kernel at p = 8) and the K steps that hold nothing but padding
// are not issued.  Each CTA loads its own 128 source rows and half of the
// offset matrix's rows; the first issues the MMAs for both.  Above 256 columns
// |j| is split into column blocks (one per grid row); where one block leaves
// room, the offset matrices of several child classes pi are stacked along N
// (one MMA of up to 256 columns), so small |j| still run the long MMAs the
// tensor pipe needs (3D Laplace p = 10: |j| = 121 -> two classes of 128
// columns).  A pair runs every (sigma, delta) that is an interaction for at
// least one of its classes; an offset that is adjacent for one class meets that
// class's zero matrix.  A launch of few tiles splits each tile's combinations
// over the pairs of a larger cluster (choose_split).
//
// Precision: TF32 (one pass), or TF32x3 / BF16x3 (a = a_hi + a_lo split,
// three passes a_hi b_hi + a_hi b_lo + a_lo b_hi), FP32 accumulation.
#include <algorithm>
#include <cstring>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "adaptive.cuh"
#include "expansions.cuh"
#include "tc_ptx.cuh"

cudaError_t launch_m2l_simt_levels(const fmm_plan_s* P, const Workspace& ws, int l0, int l1,
                                   cudaStream_t st, int* nl);

namespace {

constexpr int kBM = 128;       // target parents per CTA = TMEM lanes (the MMA's M is a pair's 256)
constexpr int kMaxN = 256;     // MMA N: columns of i (times stacked classes)
constexpr int kMaxStages = 8;  // pipeline depth bound
constexpr int kSmemCap = 227 * 1024;  // opt-in shared memory per CTA

// Operand formats: tf32 (fp32 storage, kind::tf32) and bf16 (kind::f16).  Both
// split a value into hi + lo.  The split works on the float rounding of the
// value (one conversion from FP64): lo = f - hi is exact in float, and keeps
// the bits the tf32/bf16 format drops from hi.
struct FmtTF32 {
  using T = float;
  static constexpr int kIdesc = 2;
  static constexpr bool kF16 = false;
  static constexpr bool kScaled = false;
  static constexpr CUtensorMapDataType kMapType = CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
  static __device__ __forceinline__ void split(float f, T& hi, T& lo) {
    const float h = tc::tf32_rna(f);
    hi = h;
    lo = tc::tf32_rna(f - h);
  }
};
struct FmtBF16 {
  using T = __nv_bfloat16;
  static constexpr int kIdesc = 1;
  static constexpr bool kF16 = true;
  static constexpr bool kScaled = false;
  static constexpr CUtensorMapDataType kMapType = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  static __device__ __forceinline__ void split(float f, T& hi, T& lo) {
    hi = __float2bfloat16_rn(f);
    lo = __float2bfloat16_rn(f - __bfloat162float(hi));
  }
};
// fp16 (kind::f16, type 0): tf32's 11-bit significand, a 5-bit exponent.
// The operands are scaled into its range (kScaled).  With S_m = m! (sqrt 2)^|m|
// (the float table fact_f): a box's multipole bt_q S_q, times 2^-e_box so that
// its largest entry lies in [1/2, 1); the offset matrix Ht_{i+q} / (S_i S_q)
// over the power of two of the level's derivative scale.  Dividing by i! q!
// turns the Hankel entries into binomially weighted Taylor coefficients of G,
// which grow like (sqrt 2)^{|i+q|} at the nearest offsets (their singularity
// lies sqrt 2 box sides away in complex directions); (sqrt 2)^{|i+q|} takes
// that growth out, so the entries stay below ~10 up to p = 16 (65504 is
// fp16's largest) while the rows of high |i| stay out of the subnormal range.
// The draining warps multiply each offset's product by 2^e_box of the row's
// source box and the epilogue by S_i and the table scale.
struct FmtF16 {
  using T = __half;
  static constexpr int kIdesc = 0;
  static constexpr bool kF16 = true;
  static constexpr bool kScaled = true;
  static constexpr CUtensorMapDataType kMapType = CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  static __device__ __forceinline__ void split(float f, T& hi, T& lo) {
    hi = __float2half_rn(f);
    lo = __float2half_rn(f - __half2float(hi));
  }
};

// the power of two of the derivative tables' scale at level l (Laplace
// 1/(4 pi s), biharmonic s, the screened and oscillatory kernels 1/s): the
// F16X3 offset matrices are divided by it
__host__ __device__ inline double tc_norm(int kernel, double size, int l) {
  const double s = size / (double)(1 << l);
  const double ds = kernel == FMM_KERNEL_LAPLACE ? 1.0 / (4.0 * 3.14159265358979323846 * s)
                    : kernel == FMM_KERNEL_BIHARMONIC ? s
                                                      : 1.0 / s;
  return std::ldexp(1.0, std::ilogb(ds));
}

// A pipeline stage holds one K chunk of every operand the passes read:
// [sources hi | offset matrices hi | sources lo | offset matrices lo], in
// 128-byte chunks (128-byte swizzle); the row bytes must match tc_shape().
// Each stage feeds 4 K steps (12 MMAs in the split forms) per barrier round:
// measured on GB300 (one-CTA form), 64-byte chunks (twice the rounds) ran the
// contraction 15-18% slower (biharmonic p = 8, L = 6: 11.9 against 10.1 ms, TF32x3).
template <int NPASS>
struct Cfg {
  static constexpr int kRowBytes = 128;
  static constexpr int kKSteps = kRowBytes / 32;  // MMAs of 32 bytes of K per chunk
  static constexpr int kTileS = kBM * kRowBytes;  // the source tile (MMA A)
  static constexpr int kHalves = NPASS == 1 ? 1 : 2;
  static __device__ __forceinline__ uint64_t desc(uint32_t saddr) { return tc::desc_sw128(saddr); }
  // bytes of one stage for `brows` rows of the offset matrices
  static __host__ __device__ int stage_bytes(int brows) {
    return kHalves * (kTileS + brows * kRowBytes);
  }
};

// Packed tail of the split forms.  When |j| leaves t elements over a whole
// number of K chunks and 3 t fit one chunk, the last chunk of the hi rows holds
// [a_hi | a_hi | a_lo] against [b_hi | b_lo | b_hi] (t elements each): one MMA
// per K step does the three products, and the lo rows' chunk is not loaded.
// |j| = 130 (t = 2): 25 MMAs per combination instead of 27 and a sixth less
// operand traffic.  k0: first element of the tail; t = 0: no packed tail.
struct KTail {
  int k0, t;
};
inline KTail k_tail(int nj, int row_elems, int halves) {
  const int t = nj % row_elems;
  if (halves == 2 && t > 0 && 3 * t <= row_elems) return KTail{nj - t, t};
  return KTail{1 << 30, 0};
}
// the coefficient stored at element q of a row (-1: padding); *part: the third
// of the packed tail it lies in (0 outside the tail)
__device__ __forceinline__ int row_elem(const KTail& kt, int nj, int q, int* part) {
  *part = 0;
  if (q < kt.k0) return q < nj ? q : -1;
  const int r = q - kt.k0;
  if (r >= 3 * kt.t) return -1;
  *part = r / kt.t;
  return kt.k0 + r - *part * kt.t;
}

// ---- operand packing ------------------------------------------------------
// multipoles of every level l >= 2 (lexicographic boxes, FP64, nj per box) ->
// Bpar_l[sigma][Tz][Ty][Tx][JP] (hi, and lo for the split);
// blockIdx.y = l - 2, levels stored back to back like the expansions.
struct LevOff {
  int64_t o[FMM_MAX_LEVELS + 1];
};

template <typename F>
__global__ void k_pack_beta(const double* __restrict__ mp, const LevOff lev_off, int nj, int JP,
                            const KTail kt, typename F::T* __restrict__ bhi, typename F::T* __restrict__ blo) {
  const int l = blockIdx.y + 2;
  const int nl = 1 << l, H = nl >> 1;
  const unsigned tot = (unsigned)JP << (3 * l);  // boxes of the level x JP (< 2^32)
  const double* mpl = mp + lev_off.o[l] * nj;
  typename F::T* bh = bhi + lev_off.o[l] * JP;
  typename F::T* bl = blo ? blo + lev_off.o[l] * JP : nullptr;
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += gridDim.x * blockDim.x) {
    const unsigned b = e / (unsigned)JP;  // 32-bit division (JP need not be a power of two)
    const int q = (int)(e - b * (unsigned)JP);
    const int x = (int)(b & (nl - 1)), y = (int)((b >> l) & (nl - 1)), z = (int)(b >> (2 * l));
    const int sg = (x & 1) | ((y & 1) << 1) | ((z & 1) << 2);
    const size_t dst = ((((size_t)sg * H + (z >> 1)) * H + (y >> 1)) * H + (x >> 1)) * JP + q;
    int part;
    const int qs = row_elem(kt, nj, q, &part);
    const float v = qs >= 0 ? (float)mpl[(size_t)b * nj + qs] : 0.f;
    typename F::T hi, lo;
    F::split(v, hi, lo);
    bh[dst] = part == 2 ? lo : hi;
    if (bl) bl[dst] = lo;
  }
}

// The F16X3 packing: one warp per box, bt_q S_q scaled by 2^-e so that its
// largest entry lies in [1/2, 1); 2^e goes to bscale in the same parity-split
// cell order (one value per box).
template <typename F>
__global__ void __launch_bounds__(256) k_pack_beta_scaled(const double* __restrict__ mp,
                                                          const LevOff lev_off, int nj, int JP,
                                                          const KTail kt, const float* __restrict__ fact_f,
                                                          typename F::T* __restrict__ bhi,
                                                          typename F::T* __restrict__ blo,
                                                          float* __restrict__ bscale) {
  const int l = blockIdx.y + 2;
  const int nl = 1 << l, H = nl >> 1;
  const int64_t nbox = (int64_t)1 << (3 * l);
  const double* mpl = mp + lev_off.o[l] * nj;
  typename F::T* bh = bhi + lev_off.o[l] * JP;
  typename F::T* bl = blo + lev_off.o[l] * JP;
  float* bs = bscale + lev_off.o[l];
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; b < nbox; b += nw) {
    const int x = (int)(b & (nl - 1)), y = (int)((b >> l) & (nl - 1)), z = (int)(b >> (2 * l));
    const int sg = (x & 1) | ((y & 1) << 1) | ((z & 1) << 2);
    const size_t cell = (((size_t)sg * H + (z >> 1)) * H + (y >> 1)) * H + (x >> 1);
    const double* src = mpl + b * nj;
    float m = 0.f;
    for (int q = lane; q < nj; q += 32) m = fmaxf(m, fabsf((float)src[q] * fact_f[q]));
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    const int e = m > 0.f ? ilogbf(m) + 1 : 0;
    const float down = ldexpf(1.f, -e);  // exact
    for (int q = lane; q < JP; q += 32) {
      int part;
      const int qs = row_elem(kt, nj, q, &part);
      const float v = qs >= 0 ? (float)src[qs] * fact_f[qs] * down : 0.f;
      typename F::T hi, lo;
      F::split(v, hi, lo);
      bh[cell * JP + q] = part == 2 ? lo : hi;
      bl[cell * JP + q] = lo;
    }
    if (lane == 0) bs[cell] = ldexpf(1.f, e);
  }
}

// dense offset matrices A_h[i][q] = Ht_h[i + q] (rows i < NPT, columns q < JP,
// zero outside j) for the 343 offsets of a level: one block per unsigned offset
// |h| (grid.x), table level (grid.y) and share of the rows (grid.z).  The matrix of a
// reflected offset differs by signs, (-1)^(i_k + q_k) per reflected axis, so an
// entry is formed and split once and written with its sign to up to eight
// matrices.  The offsets of adjacent boxes get zero matrices: a CTA that serves
// several child classes meets them for the classes the offset is not an
// interaction of.  No FP64 in the inner loop: F16X3's Ht_{i+q} / (S_i S_q norm) is a
// product of double-word floats whose high part is its float rounding (the FP64
// products of one block per offset took 104 us at p = 8, 50k points).
constexpr int kTmatSplit = 8;
template <typename F>
size_t tmat_smem(const PlanDev& pd, int jp) {
  const size_t nrow = (size_t)hankel_rows(pd);
  return sizeof(float2) * ((size_t)pd.nh + (F::kScaled ? pd.nj : 0)) + sizeof(int) * nrow +
         sizeof(int) * (size_t)jp;
}
__device__ __forceinline__ float flip(float v) { return -v; }
__device__ __forceinline__ __half flip(__half v) { return __hneg(v); }
__device__ __forceinline__ __nv_bfloat16 flip(__nv_bfloat16 v) { return __hneg(v); }
template <typename F>
__global__ void __launch_bounds__(256) k_build_tmat(PlanDev pd, const Geom* __restrict__ g,
                                                    const double* __restrict__ htab,
                                                    int NPT, int JP, const KTail kt,
                                                    typename F::T* __restrict__ thi,
                                                    typename F::T* __restrict__ tlo) {
  using T = typename F::T;
  struct alignas(2 * sizeof(T)) Two {
    T a, b;
  };
  htab += (size_t)blockIdx.y * 343 * pd.nh;
  thi += (size_t)blockIdx.y * 343 * NPT * JP;
  if (tlo) tlo += (size_t)blockIdx.y * 343 * NPT * JP;
  const int h[3] = {(int)blockIdx.x & 3, ((int)blockIdx.x >> 2) & 3, (int)blockIdx.x >> 4};
  const bool far = h[0] > 1 || h[1] > 1 || h[2] > 1;
  const int r0 = NPT * (int)blockIdx.z / kTmatSplit, r1 = NPT * ((int)blockIdx.z + 1) / kTmatSplit;
  const int P2 = 2 * pd.p, nrow = hankel_rows(pd);
  extern __shared__ __align__(16) unsigned char smtm[];
  float2* hv = reinterpret_cast<float2*>(smtm);  // Hankel row: (hi, lo) split, or double-word
  float2* rs = hv + pd.nh;                        // F16X3: 1 / S_m, double-word
  int* hrow = reinterpret_cast<int*>(rs + (F::kScaled ? pd.nj : 0));
  int* qmi = hrow + nrow;  // index of a column's coefficient, its tail third in bits 28..29; -1: padding
  for (int e = threadIdx.x; e < nrow; e += blockDim.x) hrow[e] = pd.hrow[e];
  __syncthreads();
  if (far) {
    const double* H = htab + (size_t)((h[0] + 3) + 7 * (h[1] + 3) + 49 * (h[2] + 3)) * pd.nh;
    const double rn = F::kScaled ? 1.0 / tc_norm(pd.kernel, g->size, blockIdx.y + 2) : 1.0;
    // F16X3: over the table's power of two; 2^(-3 |m|) here against 2^(3 |i|), 2^(3 |q|)
    // of the scalings keeps the double-word products inside the float exponents
    for (int e = threadIdx.x; e < nrow * (P2 + 1); e += blockDim.x) {
      const int row = e / (P2 + 1), m0 = e - row * (P2 + 1);
      const int deg = m0 + row % (P2 + 1) + row / (P2 + 1);
      if (deg > P2) continue;
      const int at = hrow[row] + m0;
      if (F::kScaled) {
        const dwf v = coef_in<dwf>(H[at] * rn * pow2_neg<double>(3 * deg));
        hv[at] = make_float2(v.h, v.l);
      } else {
        T vh, vl;
        F::split((float)H[at], vh, vl);
        hv[at] = make_float2((float)vh, (float)vl);
      }
    }
    if (F::kScaled)
      for (int e = threadIdx.x; e < pd.nj; e += blockDim.x) {
        // the very float the packing uses
        const dwf v = coef_in<dwf>(1.0 / ((double)pd.fact_f[e] * pow2_neg<double>(3 * pd.mi[e].w)));
        rs[e] = make_float2(v.h, v.l);
      }
    for (int e = threadIdx.x; e < JP; e += blockDim.x) {
      int part;
      const int q = row_elem(kt, pd.nj, e, &part);
      qmi[e] = q < 0 ? -1 : q | (part << 28);
    }
  }
  __syncthreads();
  // the matrices this block writes: variant bit k flips axis k (where h_k != 0)
  size_t dst[8];
  int nvar = 0, flips[8];
  for (int var = 0; var < 8; ++var) {
    if (((var & 1) && !h[0]) || ((var & 2) && !h[1]) || ((var & 4) && !h[2])) continue;
    const int o = (var & 1 ? 3 - h[0] : 3 + h[0]) + 7 * (var & 2 ? 3 - h[1] : 3 + h[1]) +
                  49 * (var & 4 ? 3 - h[2] : 3 + h[2]);
    flips[nvar] = var;
    dst[nvar++] = (size_t)o * NPT * JP;
  }
  const T zero = T(0.f);
  const int half = JP / 2, tot = (r1 - r0) * half;
  for (int e = threadIdx.x; e < tot; e += blockDim.x) {
    const int i = r0 + e / half, q2 = (e % half) * 2;
    T vh[2] = {zero, zero}, vl[2] = {zero, zero};
    int odd[2] = {0, 0};  // parities of i + q
    if (far && i < pd.nj) {
      const char4 a = pd.mi[i];
      dwf ri(1);
      if (F::kScaled) ri = dwf(rs[i].x, rs[i].y);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int w = qmi[q2 + k];
        if (w < 0) continue;
        const int q = w & 0xfffffff, part = w >> 28;
        const char4 b = pd.mi[q];
        const int m0 = a.x + b.x, m1 = a.y + b.y, m2 = a.z + b.z;
        const float2 t = hv[hrow[m2 * (P2 + 1) + m1] + m0];
        T hi, lo;
        if (F::kScaled) {
          const dwf v = dwf(t.x, t.y) * (ri * dwf(rs[q].x, rs[q].y));
          F::split(v.h, hi, lo);
        } else {
          hi = T(t.x);
          lo = T(t.y);
        }
        vh[k] = part == 1 ? lo : hi;
        vl[k] = lo;
        odd[k] = (m0 & 1) | ((m1 & 1) << 1) | ((m2 & 1) << 2);
      }
    }
    const size_t at = (size_t)i * JP + q2;
    for (int v = 0; v < nvar; ++v) {
      const bool n0 = __popc(odd[0] & flips[v]) & 1, n1 = __popc(odd[1] & flips[v]) & 1;
      *reinterpret_cast<Two*>(thi + dst[v] + at) = Two{n0 ? flip(vh[0]) : vh[0],
                                                       n1 ? flip(vh[1]) : vh[1]};
      if (tlo)
        *reinterpret_cast<Two*>(tlo + dst[v] + at) = Two{n0 ? flip(vl[0]) : vl[0],
                                                         n1 ? flip(vl[1]) : vl[1]};
    }
  }
}

// ---- the contraction --------------------------------------------------------
// CTA pairs (cta_group::2).  The two CTAs of a pair hold two neighbouring tiles
// of 128 target parents of the same child class: each loads its own 128 source
// rows and HALF of the offset matrix's rows, and one MMA of M = 256 reads both
// halves in both shared memories and fills both tensor memories.  Against one
// MMA of M = 128 per SM this halves the offset matrices' L2 and shared-memory
// traffic (133 instead of 208 KB per combination and SM for biharmonic p = 8),
// deepens the stage ring from 3 to 4 stages and halves the issue work per
// product.  N is a multiple of 32 there (130 -> 160).
//
// Warp roles: warps 0-7 drain TMEM (warp w reads TMEM lanes 32(w%4).. = target
// parents, and half of the columns), warps 8 and 11 load this CTA's source rows
// and its half of the offset matrices by TMA, warps 9 and 10 of the pair's even
// CTA (the leader) issue the MMAs of both, the even and the odd combinations.
// One issuing thread spends ~34 cycles on an MMA, ~150 on a TMA instruction and
// ~100 on each wait, in series, which alone came to 2,460 and 2,000 cycles per
// combination (F16X3, biharmonic p = 8) against 2,000 of MMA time; two of each
// overlap theirs.  The tensor cores truncate when they accumulate,
// so a long K loop in one accumulator drifts; each offset's partial product
// therefore goes to one of two 256-column TMEM buffers (the whole 512 columns),
// and the draining warps add it into float registers (round-to-nearest) while
// the MMA warp fills the other buffer.  At the end the sums go through shared
// memory so that the FP64 local expansions are written row by row (coalesced).
// A TMEM load waits its turn between MMAs, so the drain's time is set by the
// NUMBER of load instructions per SM sub-partition: with sixteen warps of
// 8-column loads (20 of them for N = 160) it took 2,870 cycles per combination
// and held the MMAs up; eight warps with 64-column loads need four.  Their
// registers (up to 128 sums and 64 columns in flight) come from the
// producers' warpgroup (setmaxnreg).
//
// Splits.  A CTA walks up to 189-216 combinations in series, so a tree with few
// tiles leaves SMs idle for the whole walk (3D Laplace p = 8, L = 4: 40 CTAs).
// There a cluster holds `split` pairs that share the tiles and each walk a part
// of the combinations; the sums meet in the epilogue through distributed shared
// memory, in rank order (the result does not depend on timing).
constexpr int kEpiWarps = 8;
constexpr int kNBuf = 2;         // accumulator buffers of 256 columns
constexpr int kTmemCols = 512;   // the whole tensor memory of the SM
constexpr int kTcThreads = (kEpiWarps + 4) * 32;
// adaptive plans: a fourth warpgroup gathers the source rows of sparse levels
constexpr int kTcThreadsA = kTcThreads + 128;
// registers per thread: 168 at launch of 384 threads (adaptive: 128 of 512); the
// draining warpgroups take what the others give up: 256 x 216 + 128 x 72 =
// 384 x 168, 256 x 192 + 256 x 64 = 512 x 128
template <bool ADAPT>
struct TcRegs {
  static constexpr int kDrain = ADAPT ? 192 : 216, kIssue = ADAPT ? 64 : 72;
};
constexpr int kMaxSplit = 4;     // pairs per cluster (8 CTAs: the portable cluster size)
constexpr int kCombos = 216;     // source children x parent shifts
// shared memory after the stages: barriers and flags, the combinations, and
// the source-cell offsets of the combinations (F16X3) or the hand-over of gathered
// rows between the CTAs of a pair (GatherCtl: adaptive trees; never both)
constexpr int kCtlBytes = 256;
constexpr int kTailBytes = kCtlBytes + 2 * kCombos * (int)sizeof(int);
// running sums per thread: half of the MMA's columns; instantiated for
// N <= 192 and N <= 256
constexpr int kColGroups = kEpiWarps / 4;
constexpr int kColsSmall = 96;
constexpr int kColsLarge = kMaxN / kColGroups;

// barrier of the draining warps alone (the TMA and MMA threads go their way)
__device__ __forceinline__ void drain_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");
}
// barrier of the CTA's threads, met from the branches of the roles
template <int THREADS>
__device__ __forceinline__ void cta_sync() {
  asm volatile("bar.sync 0, %0;" ::"n"(THREADS) : "memory");
}

// add W (16, 32, 48 or 64) TMEM columns, times rs if SCALED, to sum[0 .. W)
template <int W, bool SCALED>
__device__ __forceinline__ void drain_columns(uint32_t taddr, float rs, float* sum) {
  uint32_t r[W];
  if (W == 64) {
    tc::tmem_ld64_nowait(taddr, r);
  } else {
    if (W >= 32) tc::tmem_ld32_nowait(taddr, r);
    if (W & 16) tc::tmem_ld16_nowait(taddr + (W & 32), r + (W & 32));
  }
  tc::tmem_wait();
#pragma unroll
  for (int j = 0; j < W; ++j)
    sum[j] = SCALED ? fmaf(__uint_as_float(r[j]), rs, sum[j]) : sum[j] + __uint_as_float(r[j]);
}
// the same for w <= MOST columns (a multiple of 16)
template <bool SCALED, int MOST>
__device__ __forceinline__ void drain_upto(uint32_t taddr, int w, float rs, float* sum) {
  if (MOST >= 64 && w >= 64) drain_columns<64, SCALED>(taddr, rs, sum);
  else if (MOST >= 64 && w == 48) drain_columns<48, SCALED>(taddr, rs, sum);
  else if (w >= 32) drain_columns<32, SCALED>(taddr, rs, sum);
  else if (w == 16) drain_columns<16, SCALED>(taddr, rs, sum);
}

// Combination of a source child sigma and a parent shift delta, packed:
// sigma | (dx + 1) << 3 | (dy + 1) << 5 | (dz + 1) << 7 | h0 << 9, where h0 is
// the offset index (0..342) of the combination for targets of class 0; the
// index for class pi is h0 + class_step(pi) (h = pi - sigma - 2 delta is
// linear in pi).  A CTA lists its combinations once, in shared memory: the
// three pipeline roles then read one word per combination.  Recomputing them
// (216 candidates, div/mod chains, a loop over the classes) in the single
// issuing threads cost more than the MMAs: 4,118 cycles per combination, of
// which 350 were waits, against 3,030 with the table (one-SM MMAs, biharmonic
// p = 8, L = 6, F16X3; the contraction 6.85 -> 5.14 ms).
__device__ __forceinline__ int class_step(int pi) {
  return (pi & 1) + 7 * ((pi >> 1) & 1) + 49 * ((pi >> 2) & 1);
}
// combination c of the 216 (sigma fastest); *any: it is an interaction (not
// adjacent) for at least one of the classes pi0 .. pi0 + ncls - 1
__device__ __forceinline__ int pack_combo(int c, int pi0, int ncls, bool* any) {
  const int sg = c & 7, di = c >> 3;
  const int dx = di % 3 - 1, dy = (di / 3) % 3 - 1, dz = di / 9 - 1;
  const int hx = -(sg & 1) - 2 * dx, hy = -((sg >> 1) & 1) - 2 * dy, hz = -((sg >> 2) & 1) - 2 * dz;
  bool far = false;
  for (int pi = pi0; pi < pi0 + ncls; ++pi) {
    const int x = hx + (pi & 1), y = hy + ((pi >> 1) & 1), z = hz + ((pi >> 2) & 1);
    far |= !(x >= -1 && x <= 1 && y >= -1 && y <= 1 && z >= -1 && z <= 1);
  }
  *any = far;
  return sg | (dx + 1) << 3 | (dy + 1) << 5 | (dz + 1) << 7 |
         ((hx + 3) + 7 * (hy + 3) + 49 * (hz + 3)) << 9;
}
struct Combo {
  int sg, dx, dy, dz, h0;
};
__device__ __forceinline__ Combo unpack_combo(int v) {
  Combo k;
  k.sg = v & 7;
  k.dx = ((v >> 3) & 3) - 1;
  k.dy = ((v >> 5) & 3) - 1;
  k.dz = ((v >> 7) & 3) - 1;
  k.h0 = v >> 9;
  return k;
}

// One launch covers every level: pairs [first_pair, ...) belong to level l
// (pair = tile pair * (8 / ncls) + class group), grid.y = column block of i;
// grid.x holds 2 * split CTAs per pair, one cluster.
// The parent grid of a level is Hx x Hy x Hz cells: the whole level of a
// uniform tree (Hx = Hy = Hz = 2^(l-1), boxes lexicographic), or, for an
// adaptive tree, the window of parents spanned by the level's boxes, with
// map[(pi, cell)] the box at that position (-1: none).
// A homogeneous kernel shares one set of offset matrices over the levels, so a
// small level can ride along in the pairs of a level of one tile: the odd CTA
// takes its whole parent grid (H2^3 parents, H2 = 2^(l2-1); l2 = 0: none).
// This keeps the tiny coarse levels from forming a wave of their own.
// Gathered levels (adaptive trees, gather != 0): the MMA's rows are target
// cells of one class taken from a list (tlist: the cells holding a box with
// targets, grouped by class at offsets toff[0..8], Morton order inside a
// class), and each offset's source rows are gathered from the parity-split
// window (rows ghi, glo; row zero_row is all zeros and stands for a source
// outside the window) by four warps' cp.async copies into the layout the TMA
// would have written.  Pair 8k + u of the level takes entries
// 256k .. 256k + 255 of class u's list, 128 per CTA: the k-th chunks of the
// eight classes cover about the same region and run together, so the window
// rows they share are read from L2 (class-major order measured 2.7x slower per
// CTA, the window exceeding L2); pairs past a class's list leave at once.
struct TcLevel {
  CUtensorMap S, Slo;    // parity-split multipoles of the level (MMA A)
  CUtensorMap S2, S2lo;  // multipoles of the riding level l2
  CUtensorMap H, Hlo;    // offset matrices of the level (MMA B)
  double* lc;            // local expansions (level base, or all boxes with map)
  double* lc2;           // local expansions of level l2 (base)
  const int* map;        // adaptive: window cell -> box; null for uniform levels
  const float* bscale;   // F16X3: 2^e_box of the level's packed multipoles (cell order)
  const float* bscale2;  // the same for the riding level l2
  const int* tlist;      // gathered levels: target cells grouped by class
  const int* toff;       // gathered levels: offsets of the classes in tlist [9]
  const char* ghi;       // gathered levels: the window's rows (hi, lo), JP per row
  const char* glo;
  float scale, scale2;   // exact powers of two (shared offset matrices)
  int l, BX, BY, BZ, ntx, nty, ntiles, first_pair, Hx, Hy, Hz;
  int l2;
  int gather, zero_row;
};
constexpr int kTcMaxLevels = 10;
struct TcParams {
  TcLevel lev[kTcMaxLevels];
  int nlev, nj, jchunks, ksteps_last;
  int packed;          // the last K chunk is a packed tail (KTail): hi rows only, one MMA a step
  int nc, npt, ncls;   // columns per block, rows per offset matrix, stacked classes
  int nmma, hb_n, hb_rows;  // MMA N; a CTA's half of B: boxes and rows of each
  int split;           // pairs per cluster
  int nstages, stage_bytes;
  long long wait_cycles;  // limit of the pipeline's mbarrier waits
  int* err;
  // F16X3: the table norm (tc_norm at table level tlev_fixed, or at the CTA's
  // level when 0) and m! of the local coefficients
  const Geom* geom;
  int kernel, tlev_fixed;
  const float* fact_f;
};

// The tile of target parents one CTA holds: n rows (parents, x fastest inside
// BX x BY x BZ from X0, Y0, Z0) of a grid Hx x Hy x Hz of level l.
struct TcTile {
  int n, X0, Y0, Z0, BX, BY, Hx, Hy, Hz, l;
};
__device__ __forceinline__ TcTile tile_of(const TcLevel& LV, int tp, int half) {
  TcTile t;
  if (half && LV.l2) {  // the riding level (its host level has one tile)
    const int H2 = 1 << (LV.l2 - 1);
    t.n = H2 * H2 * H2;
    t.X0 = t.Y0 = t.Z0 = 0;
    t.BX = t.BY = t.Hx = t.Hy = t.Hz = H2;
    t.l = LV.l2;
    return t;
  }
  const int tile = 2 * tp + half;
  t.n = tile < LV.ntiles ? LV.BX * LV.BY * LV.BZ : 0;
  t.X0 = tile % LV.ntx * LV.BX;
  t.Y0 = tile / LV.ntx % LV.nty * LV.BY;
  t.Z0 = tile / (LV.ntx * LV.nty) * LV.BZ;
  t.BX = LV.BX;
  t.BY = LV.BY;
  t.Hx = LV.Hx;
  t.Hy = LV.Hy;
  t.Hz = LV.Hz;
  t.l = LV.l;
  return t;
}

// F16X3: where the scale 2^e_box of the source box feeding TMEM lane `row`
// is found, packed in one register (the drain has none to spare): the row's
// parent (x, y, z) gives base = (z Hy + y) Hx + x (< 2^21 for levels <= 8),
// bits 21..26 flag the neighbours that exist (x-1, x+1, y-1, y+1, z-1, z+1)
// and bit 27 a row inside the grid (0: no source).
__device__ __forceinline__ int row_scale_setup(const TcTile& t, int row) {
  if (row >= t.n) return 0;
  const int x = t.X0 + row % t.BX, y = t.Y0 + row / t.BX % t.BY, z = t.Z0 + row / (t.BX * t.BY);
  if (x >= t.Hx || y >= t.Hy || z >= t.Hz) return 0;  // a target outside the grid: not stored
  const int mask = (x > 0) | ((x + 1 < t.Hx) << 1) | ((y > 0) << 2) | ((y + 1 < t.Hy) << 3) |
                   ((z > 0) << 4) | ((z + 1 < t.Hz) << 5) | (1 << 6);
  return ((z * t.Hy + y) * t.Hx + x) | (mask << 21);
}

// 2^e_box of the source (combination k, whose cell lies `so` cells from the
// target's); 0 for a source outside the grid, whose TMA rows are zero
__device__ __forceinline__ float row_scale(const float* __restrict__ bs, int rb, const Combo& k,
                                           int so) {
  const int mask = rb >> 21;
  const bool ok = (mask & 64) && (k.dx >= 0 || (mask & 1)) && (k.dx <= 0 || (mask & 2)) &&
                  (k.dy >= 0 || (mask & 4)) && (k.dy <= 0 || (mask & 8)) &&
                  (k.dz >= 0 || (mask & 16)) && (k.dz <= 0 || (mask & 32));
  return ok ? bs[(rb & 0x1fffff) + so] : 0.f;
}

// pipeline wait: the default bounded wait, or (SHORTW, the instantiation that
// tests run with a shortened limit) the polling wait of mbar_wait_short;
// CLUSTER: acquiring what another CTA wrote to its shared memory
template <bool SHORTW, bool CLUSTER = false>
__device__ __forceinline__ bool pwait(uint64_t* bar, uint32_t parity, int* err, long long lim) {
  return SHORTW ? tc::mbar_wait_short<CLUSTER>(bar, parity, err, lim)
                : tc::mbar_wait<CLUSTER>(bar, parity, err);
}
// bounded wait without an error report (the waits before a CTA leaves)
__device__ __forceinline__ void settle(uint64_t* bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!tc::mbar_try_wait(bar, parity) && clock64() - t0 < tc::kWaitCycles) {
  }
}

// barriers and flags of a CTA (after the stages; the same offset in every CTA)
struct TcCtl {
  uint64_t full[kMaxStages];   // stage filled: the leader's counts both CTAs' loads
  uint64_t empty[kMaxStages];  // stage consumed (MMA commit, to both CTAs)
  uint64_t accf[kNBuf];        // accumulator filled (MMA commit, to both CTAs)
  uint64_t acce[kNBuf];        // accumulator drained (the leader's: both CTAs' warps)
  uint64_t drainb;             // all MMAs of the pair finished (leader)
  uint64_t turn[2];            // leader: issuing warp w may wait for its next stages
  uint32_t tslot;
  float tn;                    // F16X3: the table norm of the offset matrices
  int bad;                     // a role of this CTA gave up
  int ncombos;
  int armed[2];   // stage rounds whose source rows / offset matrices were requested
  int gathered[4];  // gathered levels, per gathering warp: rounds reported filled
  // leader, per issuing warp w (combinations g = w, w + 2, ...): the offsets whose
  // accumulator was committed, and the chunks committed of the next one
  int accs[2], part[2];
};
static_assert(sizeof(TcCtl) <= kCtlBytes, "control block");

// Gathered levels.  The odd CTA's rows are written by its own threads and read by
// MMAs that the leader issues, so they have to be published at cluster scope.  A
// release at that scope takes one to two thousand cycles beside the copies in
// flight, more than a round, so three warps that have nothing else to do there
// relay every third round each: the gathering warps arrive on `rows` (CTA
// scope), the relay on the leader's `peer` (release, cluster), where one
// warp receives (acquire, cluster) and arrives on `full` for the issuers.  2M
// and 60k points: 11,605 and 1,074 us a step; with the release in the gathering
// warps' own arrivals 15,222 and 1,437.
constexpr int kRelays = 3;  // warps kEpiWarps .. kEpiWarps + 2 of the odd CTA
struct GatherCtl {
  uint64_t rows[kMaxStages];  // odd CTA: rows of the stage written
  uint64_t peer[kMaxStages];  // leader: the odd CTA's rows published
  int received;               // leader: rounds handed on to `full`
};
static_assert(sizeof(GatherCtl) <= kCombos * sizeof(int), "hand-over block");

// Before a CTA leaves (after a cluster barrier, so the counters are final):
// wait, bounded, until every copy into its stages has landed and every commit
// aimed at its barriers has arrived.  When nothing went wrong all of it has
// happened and the waits return at once.  After a timeout the loaders of a pair
// may have stopped at different rounds: the leader then settles, on its
// barriers, the bytes and the arrivals of gathered rows that will not come, and
// arms the rounds that only others have loaded.  srow / brow: bytes that TMA
// brings of the source rows of the leader and of the other CTA, and of one half
// of B, per stage round; a packed tail's round brings one half of them (tdiv).
__device__ __forceinline__ void close_pipeline(TcCtl* ctl, int half, uint32_t peer, int ns,
                                               bool gather, int received, const int* srow,
                                               int brow, int tdiv, int jchunks) {
  auto theirs = [&](int* p) { return tc::ld_cluster_s32(tc::map_rank(tc::smem_u32(p), peer)); };
  auto leads = [&](int* p) { return half ? theirs(p) : *p; };
  if (half == 0) {  // all loads of the pair complete on the leader's barriers
    const int n[4] = {gather ? ctl->armed[1] : ctl->armed[0], ctl->armed[1],
                      gather ? theirs(&ctl->armed[1]) : theirs(&ctl->armed[0]),
                      theirs(&ctl->armed[1])};
    int from = min(min(n[0], n[1]), min(n[2], n[3]));
    int upto = max(max(n[0], n[1]), max(n[2], n[3]));
    if (gather) {
      from = min(from, received);
      upto = max(upto, received);
      for (int k = 0; k < 4; ++k) {
        from = min(from, ctl->gathered[k]);
        upto = max(upto, ctl->gathered[k]);
      }
    }
    for (int j = from; j < upto; ++j) {
      const int by[4] = {srow[0], brow, srow[1], brow};
      int all = 0, come = 0;
      for (int k = 0; k < 4; ++k) {
        const int b = (j + 1) % jchunks ? by[k] : by[k] / tdiv;
        all += b;
        come += j < n[k] ? b : 0;
      }
      if (j >= n[0]) tc::mbar_expect_tx(&ctl->full[j % ns], (uint32_t)come);
      else if (come < all) tc::mbar_complete_tx(&ctl->full[j % ns], (uint32_t)(all - come));
      if (gather) {
        if (j >= received) tc::mbar_arrive(&ctl->full[j % ns]);
        for (int k = 0; k < 4; ++k)
          if (j >= ctl->gathered[k]) tc::mbar_arrive(&ctl->full[j % ns]);
      }
    }
    for (int j = max(0, upto - ns); j < upto; ++j)
      settle(&ctl->full[j % ns], (uint32_t)(j / ns) & 1u);
  }
  // commits: earlier rounds' have been waited for by this CTA's loaders
  int accs[2], part[2];
  for (int w = 0; w < 2; ++w) {
    accs[w] = leads(&ctl->accs[w]);
    part[w] = leads(&ctl->part[w]);
    if (accs[w] > 0) settle(&ctl->accf[w], (uint32_t)(accs[w] - 1) & 1u);
  }
  const int first = max(0, (gather ? ctl->armed[1] : min(ctl->armed[0], ctl->armed[1])) - ns);
  for (int j = first; j < first + 3 * ns; ++j) {
    const int g = j / jchunks, w = g & 1, n = g >> 1;
    if (n < accs[w] || (n == accs[w] && j - g * jchunks < part[w]))
      settle(&ctl->empty[j % ns], (uint32_t)(j / ns) & 1u);
  }
}

template <typename F, int NPASS, bool SHORTW, int NCOL, bool ADAPT>
__global__ void __launch_bounds__(ADAPT ? kTcThreadsA : kTcThreads, 1)
    k_m2l_tc(const __grid_constant__ TcParams prm) {
  using C = Cfg<NPASS>;
  constexpr int kThreads = ADAPT ? kTcThreadsA : kTcThreads;
  // the CTA's place: cluster of `split` pairs; pair `sp`, half of it
  const uint32_t crank = tc::cluster_ctarank(), leader = crank & ~1u, peer = crank ^ 1u;
  const int half = (int)(crank & 1u), sp = (int)(crank >> 1), split = prm.split;
  const int pair = (int)blockIdx.x / (2 * split);
  int li = 0;
  while (li + 1 < prm.nlev && pair >= prm.lev[li + 1].first_pair) ++li;
  const TcLevel& LV = prm.lev[li];
  const int nj = prm.nj, jchunks = prm.jchunks;
  const int nc = prm.nc, npt = prm.npt, ncls = prm.ncls;
  const int nmma = prm.nmma;  // MMA N
  const int ns = prm.nstages, sbytes = prm.stage_bytes;
  const int btile = prm.hb_n * prm.hb_rows * C::kRowBytes;  // B bytes of one stage half
  int* __restrict__ err = prm.err;
  const long long wlim = prm.wait_cycles;
  extern __shared__ __align__(1024) unsigned char smraw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smraw) + 1023) & ~(uintptr_t)1023);
  TcCtl* ctl = reinterpret_cast<TcCtl*>(sm + ns * sbytes);
  int* ctab = reinterpret_cast<int*>(sm + ns * sbytes + kCtlBytes);  // [kCombos]
  int* soff = ctab + kCombos;   // [kCombos] F16X3: source cell - target cell
  GatherCtl* gctl = reinterpret_cast<GatherCtl*>(soff);
  static_assert(!(ADAPT && F::kScaled), "soff and the hand-over block share their place");

  // the same for all lanes, and known to be: the role branches stay uniform
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int lane = threadIdx.x & 31;
  const int lb = pair - LV.first_pair;
  const int ngrp = 8 / ncls;
  const int pi0 = (lb % ngrp) * ncls;  // classes pi0 .. pi0 + ncls - 1
  const int tp = lb / ngrp;            // tile pair (gathered: chunk of the class's list)
  const bool gather = ADAPT && LV.gather;  // (ncls == 1)
  int gstart = 0, grows = 0;           // gathered levels: this CTA's entries of tlist
  if (gather) {
    const int n = LV.toff[pi0 + 1] - LV.toff[pi0], k0 = tp * 2 * kBM;
    if (k0 >= n) return;  // a surplus pair: uniform over the cluster, before any barrier or TMEM
    gstart = LV.toff[pi0] + k0 + half * kBM;
    grows = max(0, min(kBM, n - k0 - half * kBM));
  }
  const int cb = blockIdx.y;  // column block
  const TcTile tile = tile_of(LV, gather ? 0 : tp, half);

  if (LV.map && !gather) {  // a window's tile pair whose target cells hold no box: nothing to do
    int any = 0;
    for (int h = 0; h < 2; ++h) {
      const TcTile t = tile_of(LV, tp, h);
      for (int e = threadIdx.x; e < t.n * ncls; e += blockDim.x) {
        const int n = e % t.n, u = e / t.n;
        const int x = t.X0 + n % t.BX, y = t.Y0 + n / t.BX % t.BY, z = t.Z0 + n / (t.BX * t.BY);
        if (x < t.Hx && y < t.Hy && z < t.Hz)
          any |= LV.map[(((size_t)(pi0 + u) * t.Hz + z) * t.Hy + y) * t.Hx + x] >= 0;
      }
    }
    if (!__syncthreads_or(any)) return;  // uniform over the cluster, before any barrier or TMEM
  }

  if (threadIdx.x == 0) {
    // the leader's stage barriers: its loader's arrival, and (gathered rows) those of its
    // gathering warps and of the warp that receives the other CTA's
    for (int s = 0; s < ns; ++s) {
      tc::mbar_init(&ctl->full[s], gather ? 1u + 4u + 1u : 1u);
      tc::mbar_init(&ctl->empty[s], 1);
      if (gather) {
        tc::mbar_init(&gctl->rows[s], 4);
        tc::mbar_init(&gctl->peer[s], 1);
      }
    }
    if (gather) gctl->received = 0;
    for (int bf = 0; bf < kNBuf; ++bf) {
      tc::mbar_init(&ctl->accf[bf], 1);
      tc::mbar_init(&ctl->acce[bf], 2 * kEpiWarps);
    }
    tc::mbar_init(&ctl->drainb, 2);
    for (int w = 0; w < 2; ++w) tc::mbar_init(&ctl->turn[w], 1);
    ctl->bad = 0;
    for (int k = 0; k < 4; ++k) ctl->gathered[k] = 0;
    ctl->tn = F::kScaled ? (float)tc_norm(prm.kernel, prm.geom->size,
                                          prm.tlev_fixed ? prm.tlev_fixed : LV.l)
                         : 1.f;
    for (int w = 0; w < 2; ++w) ctl->armed[w] = ctl->accs[w] = ctl->part[w] = 0;
    tc::fence_mbar_init();
  }
  if (warp == 0) tc::tmem_alloc_pair(&ctl->tslot, kTmemCols);
  if (warp == 1) {  // the combinations of these classes, in order
    int n = 0;
    for (int c0 = 0; c0 < kCombos; c0 += 32) {
      bool any = false;
      const int c = c0 + lane;
      const int v = c < kCombos ? pack_combo(c, pi0, ncls, &any) : 0;
      const unsigned m = __ballot_sync(0xffffffffu, any);
      if (any) {
        const int at = n + __popc(m & ((1u << lane) - 1u));
        ctab[at] = v;
        if (F::kScaled) {
          const Combo k = unpack_combo(v);
          soff[at] = ((k.sg * tile.Hz + k.dz) * tile.Hy + k.dy) * tile.Hx + k.dx;
        }
      }
      n += __popc(m);
    }
    if (lane == 0) ctl->ncombos = n;
  }

  tc::fence_before();
  __syncthreads();
  tc::cluster_sync();  // the barriers of both CTAs are set up before any remote arrival
  tc::fence_after();
  const uint32_t tmem = ctl->tslot;
  const int c_lo = ctl->ncombos * sp / split;              // this pair's share
  const int nco = ctl->ncombos * (sp + 1) / split - c_lo;  // of the combinations
  const int* __restrict__ ct = ctab + c_lo;
  // bytes of a stage round: source rows of the leader and of the other CTA, and
  // one CTA's half of B (packed tail: the hi rows alone)
  const int srow[2] = {gather ? 0 : C::kHalves * C::kRowBytes * tile_of(LV, tp, 0).n,
                       gather ? 0 : C::kHalves * C::kRowBytes * tile_of(LV, tp, 1).n};
  const int brow = C::kHalves * btile, tdiv = prm.packed ? C::kHalves : 1;

  if (warp >= kEpiWarps) tc::regs_dec<TcRegs<ADAPT>::kIssue>();
  if (ADAPT && gather && warp >= kEpiWarps + 4) {
    // ---------------- gathered source rows ----------------
    // Warp k of four copies rows 32k .. 32k + 31 of each stage with cp.async, 16
    // bytes at a time, into the 128-byte-swizzled layout (lane i: 16-byte column
    // i % 8 of rows i / 8 + 4m): the eight addresses of a lane are computed once
    // per combination and advance by the chunk.  A round is reported one or two
    // rounds later, when its copies have landed and been ordered before the
    // MMAs' reads.  (One warp, recomputing each row's address
    // per copy, took 17,900 cycles per combination.)
    const int gw = warp - (kEpiWarps + 4);
    const int64_t pitch = (int64_t)jchunks * C::kRowBytes;  // bytes per window row
    const int Hx = LV.Hx, Hy = LV.Hy, Hz = LV.Hz;
    const int q16 = lane & 7, r0 = lane >> 3;
    int cell[8];
    uint32_t mask[2] = {0, 0};  // 7 bits per row: target present, neighbours in the window
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int n = 32 * gw + r0 + 4 * m;
      cell[m] = 0;
      if (n < grows) {
        const int c = LV.tlist[gstart + n];
        const int x = c % Hx, y = c / Hx % Hy, z = c / (Hx * Hy);
        cell[m] = c;
        const uint32_t f = 64u | (x > 0) | ((x + 1 < Hx) << 1) | ((y > 0) << 2) |
                           ((y + 1 < Hy) << 3) | ((z > 0) << 4) | ((z + 1 < Hz) << 5);
        mask[m >> 2] |= f << (7 * (m & 3));
      }
    }
    uint64_t* told_bar = half ? gctl->rows : ctl->full;
    const uint32_t dst0 = tc::smem_u32(sm) + (uint32_t)((32 * gw + r0) * C::kRowBytes);
    const uint32_t sw0 = (uint32_t)(q16 ^ r0) << 4, sw1 = (uint32_t)(q16 ^ (r0 + 4)) << 4;
    const int64_t lo_step = LV.glo - LV.ghi;
    // rounds in flight behind the current one (stages >= 3): a second one helps where the
    // ring has room for it (60k points, five stages or more: 1,074 us, 1,088 with one) and
    // holds a ring of four up (2M points: 13,075, 11,605 with one)
    const int lag = ns > 4 ? 2 : 1;
    int s = 0, kk = 0, told = 0, ts = 0;
    uint32_t ph = 0;
    uint32_t st = 0;  // stage offset
    auto tell = [&]() {  // report round `told` to this CTA's barrier
      tc::fence_proxy_async();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&told_bar[ts]);
      ++told;
      if (++ts == ns) ts = 0;
    };
    bool ok = true;
    for (int g = 0; g < nco && ok; ++g) {
      const Combo k = unpack_combo(ct[g]);
      const int step = ((k.sg * Hz + k.dz) * Hy + k.dy) * Hx + k.dx;
      const uint32_t need = 64u | (k.dx < 0) | ((k.dx > 0) << 1) | ((k.dy < 0) << 2) |
                            ((k.dy > 0) << 3) | ((k.dz < 0) << 4) | ((k.dz > 0) << 5);
      const char* src[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const bool in = ((mask[m >> 2] >> (7 * (m & 3))) & need) == need;
        src[m] = LV.ghi + (int64_t)(in ? cell[m] + step : LV.zero_row) * pitch + q16 * 16;
      }
      for (int ch = 0; ch < jchunks; ++ch, ++kk) {
        if (kk >= ns && !pwait<SHORTW>(&ctl->empty[s], ph ^ 1u, err, wlim)) {
          ok = false;
          break;
        }
        const bool both = C::kHalves == 2 && !(prm.packed && ch == jchunks - 1);
#pragma unroll
        for (int m = 0; m < 8; ++m) {
          const uint32_t d = dst0 + st + (uint32_t)(4 * m * C::kRowBytes) + (m & 1 ? sw1 : sw0);
          tc::cp_async16(d, src[m]);
          if (both) tc::cp_async16(d + (uint32_t)(C::kTileS + btile), src[m] + lo_step);
          src[m] += C::kRowBytes;
        }
        tc::cp_async_commit();
        if (kk >= lag) {
          if (lag == 2) tc::cp_async_wait<2>();
          else tc::cp_async_wait<1>();
          tell();
        }
        if (++s == ns) {
          s = 0;
          ph ^= 1u;
          st = 0;
        } else {
          st += (uint32_t)sbytes;
        }
      }
    }
    tc::cp_async_wait<0>();  // every copy of this warp has landed before it leaves
    while (told < kk) tell();
    if (lane == 0) {
      ctl->gathered[gw] = told;
      if (!ok) ctl->bad = 1;
    }
  } else if (ADAPT && gather && (half ? warp < kEpiWarps + kRelays : warp == kEpiWarps) &&
             warp >= kEpiWarps) {
    // ---------------- hand-over of the odd CTA's gathered rows ----------------
    const int first = half ? warp - kEpiWarps : 0, step = half ? kRelays : 1;
    const uint32_t lpeer = tc::map_rank(tc::smem_u32(&gctl->peer[0]), leader);
    bool ok = true;
    int kk = first, s = first % ns;
    uint32_t ph = (uint32_t)(first / ns) & 1u;
    for (; kk < nco * jchunks; kk += step) {
      ok = half ? pwait<SHORTW>(&gctl->rows[s], ph, err, wlim)
                : pwait<SHORTW, true>(&gctl->peer[s], ph, err, wlim);
      if (!ok) break;
      if (lane == 0) {
        if (half) tc::mbar_arrive_cluster_release(lpeer + 8u * (uint32_t)s);
        else tc::mbar_arrive(&ctl->full[s]);
      }
      __syncwarp();
      for (s += step; s >= ns; s -= ns) ph ^= 1u;
    }
    if (lane == 0) {
      if (!half) gctl->received = kk;
      if (!ok) ctl->bad = 1;
    }
  } else if ((warp == kEpiWarps && !gather) || warp == kEpiWarps + 3) {
    // ---------------- TMA producers ----------------
    // The whole warp walks the loop (its addresses and coordinates are then
    // uniform values, as the TMA instruction wants them) and one elected lane
    // issues.  Stage s and the parity ph of its current round advance
    // together (no division in the loop); a stage is refilled once its
    // previous round's MMAs have committed.  Both CTAs' bytes complete on the
    // leader's barrier.
    const bool lead = tc::elect_one();
    const bool rows = warp == kEpiWarps;  // source rows, or offset matrices
    const uint32_t tx = (uint32_t)(srow[0] + srow[1] + 2 * brow);
    constexpr int kElems = C::kRowBytes / (int)sizeof(typename F::T);
    const bool ride = half && LV.l2;
    const CUtensorMap* mS[2] = {ride ? &LV.S2 : &LV.S, ride ? &LV.S2lo : &LV.Slo};
    const CUtensorMap* mH[2] = {&LV.H, &LV.Hlo};
    const uint32_t lfull = tc::map_rank(tc::smem_u32(&ctl->full[0]), leader);
    const int hb_n = prm.hb_n, hb_rows = prm.hb_rows;
    int s = 0, kk = 0;
    uint32_t ph = 0;
    unsigned char* st = sm;
    bool ok = true;
    for (int g = 0; g < nco && ok; ++g) {
      const Combo k = unpack_combo(ct[g]);
      for (int ch = 0; ch < jchunks; ++ch, ++kk) {
        const bool tail = prm.packed && ch == jchunks - 1;
        if (kk >= ns && !pwait<SHORTW>(&ctl->empty[s], ph ^ 1u, err, wlim)) {
          ok = false;
          break;
        }
        if (lead) {
          const uint32_t bar = lfull + 8u * (uint32_t)s;
          const int kc = ch * kElems;  // element offset of this K chunk
          // armed by the leader's source rows' loader (gathered: its offset matrices')
          if (half == 0 && rows != gather)
            tc::mbar_expect_tx(&ctl->full[s], tail ? tx / C::kHalves : tx);
          if (rows) {
            if (tile.n) {
#pragma unroll
              for (int hf = 0; hf < C::kHalves; ++hf)
                if (!(hf && tail))
                  tc::tma_load_5d_pair(st + hf * (C::kTileS + btile), mS[hf], bar, kc,
                                       tile.X0 + k.dx, tile.Y0 + k.dy, tile.Z0 + k.dz, k.sg);
            }
          } else {
            for (int u = 0; u < hb_n; ++u) {  // this CTA's half of B's rows
              const int row = ncls == 1 ? (k.h0 + class_step(pi0)) * npt + cb * nc + half * hb_rows
                                        : (k.h0 + class_step(pi0 + half * hb_n + u)) * npt;
#pragma unroll
              for (int hf = 0; hf < C::kHalves; ++hf)
                if (!(hf && tail))
                  tc::tma_load_2d_pair(st + hf * (C::kTileS + btile) + C::kTileS +
                                           u * hb_rows * C::kRowBytes,
                                       mH[hf], bar, kc, row);
            }
          }
        }
        __syncwarp();
        if (++s == ns) {
          s = 0;
          ph ^= 1u;
          st = sm;
        } else {
          st += sbytes;
        }
      }
    }
    if (lead) {
      ctl->armed[rows ? 0 : 1] = kk;
      if (!ok) ctl->bad = 1;
    }
  } else if ((warp == kEpiWarps + 1 || warp == kEpiWarps + 2) && !half) {
    // ---------------- leader: MMA issuers ----------------
    // as above: the warp walks, one elected lane issues.  Warp w issues the
    // combinations g = w, w + 2, .. into accumulator w (its (g >> 1)-th use);
    // everything between two MMAs is kept to a few adds.  A parity wait is
    // sound one phase ahead only, so a warp waits for its stages once the other
    // has seen all stages of the combination before (its turn).
    const bool lead = tc::elect_one();
    const int w = warp - (kEpiWarps + 1);
    const uint32_t id = tc::idesc(F::kIdesc, 2 * kBM, nmma);
    const uint64_t d0 = C::desc(tc::smem_u32(sm));
    const uint64_t ob = (uint64_t)(C::kTileS >> 4);
    const uint64_t oalo = (uint64_t)((C::kTileS + btile) >> 4);
    const uint64_t oblo = (uint64_t)((2 * C::kTileS + btile) >> 4);
    const uint64_t dstep = (uint64_t)(sbytes >> 4);
    const int kl = prm.ksteps_last;
    const uint16_t both = (uint16_t)(3u << leader);
    const uint32_t dacc = tmem + (uint32_t)(w * kMaxN);
    int s = 0, part = 0;
    uint32_t ph = 0;
    auto skip = [&]() {  // the rounds of the other warp's combination
      for (s += jchunks; s >= ns; s -= ns) ph ^= 1u;
    };
    if (w) skip();
    int g = w;
    bool ok = true;
    for (; g < nco; g += 2) {
      if (g >= 2 && !pwait<SHORTW>(&ctl->acce[w], ((g >> 1) - 1) & 1, err, wlim)) {
        ok = false;  // the buffer's previous offset has not been drained
        break;
      }
      if (g >= 1 && !pwait<SHORTW>(&ctl->turn[w], ((g - 1) >> 1) & 1, err, wlim)) {
        ok = false;
        break;
      }
      for (int ch = 0; ch < jchunks; ++ch) {
        if (!pwait<SHORTW>(&ctl->full[s], ph, err, wlim)) {
          ok = false;
          part = ch;
          break;
        }
        tc::fence_after();
        if (lead) {
          if (ch == jchunks - 1) tc::mbar_arrive(&ctl->turn[w ^ 1]);
          const uint64_t da = d0 + (uint64_t)s * dstep;
          const bool last = ch == jchunks - 1;
          const bool tail = last && prm.packed;
          const int nk = last ? kl : C::kKSteps;
#pragma unroll
          for (int ks = 0; ks < C::kKSteps; ++ks) {
            if (ks < nk) {
              // one MMA consumes 32 bytes of K (8 tf32 or 16 bf16) inside the swizzle atom
              const uint64_t a = da + (uint64_t)(ks * 2);
              const uint32_t acc = (ch | ks) != 0;
              if (F::kF16) {
                tc::mma_f16_pair(dacc, a, a + ob, id, acc);
                if (NPASS == 3 && !tail) {
                  tc::mma_f16_pair(dacc, a, a + oblo, id, 1);
                  tc::mma_f16_pair(dacc, a + oalo, a + ob, id, 1);
                }
              } else {
                tc::mma_tf32_pair(dacc, a, a + ob, id, acc);
                if (NPASS == 3 && !tail) {
                  tc::mma_tf32_pair(dacc, a, a + oblo, id, 1);
                  tc::mma_tf32_pair(dacc, a + oalo, a + ob, id, 1);
                }
              }
            }
          }
          tc::mma_commit_pair(&ctl->empty[s], both);
          if (last) tc::mma_commit_pair(&ctl->accf[w], both);
        }
        __syncwarp();
        if (++s == ns) {
          s = 0;
          ph ^= 1u;
        }
      }
      if (!ok) break;
      skip();
    }
    // the commit arrives once every MMA issued so far has finished; waiting
    // for it (time-bounded, also on the error path) means TMEM is never freed
    // under a running MMA
    if (lead) {
      tc::mma_commit_pair(&ctl->drainb, (uint16_t)(1u << leader));
      ctl->accs[w] = g >> 1;  // g = w + 2 x the offsets committed
      ctl->part[w] = part;
      if (!ok) ctl->bad = 1;
    }
    settle(&ctl->drainb, 0);
  }
  if (warp >= kEpiWarps) {
    __syncwarp();
    tc::fence_before();
    cta_sync<kThreads>();
    tc::cluster_sync();
    if (threadIdx.x == kEpiWarps * 32)
      close_pipeline(ctl, half, peer, ns, gather, gather ? gctl->received : 0, srow, brow, tdiv,
                     jchunks);
    __syncwarp();
    cta_sync<kThreads>();
    tc::cluster_sync();
    return;
  }

  // ---------------- drain TMEM into float registers ----------------
  tc::regs_inc<TcRegs<ADAPT>::kDrain>();
  {
    const int quad = warp & 3;
    const int cw = nmma / kColGroups;  // columns of this warp (a multiple of 16)
    const int c0 = (warp >> 2) * cw;
    float sum[NCOL];
#pragma unroll
    for (int j = 0; j < NCOL; ++j) sum[j] = 0.f;
    bool ok = true;
    const int row = quad * 32 + lane;  // this thread's TMEM lane
    const int rb = F::kScaled ? row_scale_setup(tile, row) : 0;
    const float* __restrict__ bs = half && LV.l2 ? LV.bscale2 : LV.bscale;
    const uint32_t lacce = tc::map_rank(tc::smem_u32(&ctl->acce[0]), leader);
    for (int g = 0; g < nco; ++g) {
      const int bf = g & 1;
      // F16X3: the power of two the row's source multipole was divided by
      // (read before the wait, off the critical path)
      const float rs = F::kScaled ? row_scale(bs, rb, unpack_combo(ct[g]), soff[c_lo + g]) : 1.f;
      if (!pwait<SHORTW>(&ctl->accf[bf], (g >> 1) & 1, err, wlim)) {
        ok = false;
        break;
      }
      tc::fence_after();
      const uint32_t base =
          tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(bf * kMaxN + c0);
      // columns in flight at a time (registers)
      constexpr int kPiece = ADAPT && NCOL > 96 ? 32 : 64;
#pragma unroll
      for (int c = 0; c < NCOL; c += kPiece)
        if (c < cw) drain_upto<F::kScaled, kPiece>(base + c, cw - c, rs, sum + c);
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive_cluster(lacce + 8u * (uint32_t)bf);
    }
    // every draining warp passes the barrier below, whatever its status, so
    // that none waits for a warp that left
    if (!ok || (*(volatile int*)err & 2)) atomicOr(&ctl->bad, 1);
    drain_sync();
    if (*(volatile int*)&ctl->bad == 0) {
      // every MMA has finished and every TMA copy has been consumed: the stage
      // memory is free for the staging of the sums, [row][column] with an odd
      // pitch (the 32 lanes of a warp write 32 rows of one column)
      float* stg = reinterpret_cast<float*>(sm);
#pragma unroll
      for (int j = 0; j < NCOL; ++j)
        if (j < cw) stg[row * (nmma + 1) + c0 + j] = sum[j];
    }
  }
  __syncwarp();
  tc::fence_before();
  cta_sync<kThreads>();
  tc::cluster_sync();  // counters, flags and staged sums of the whole cluster are final
  tc::fence_after();
  // the decision to write is taken from the flags of all CTAs, the same for all
  bool good = true;
  for (int r = 0; r < 2 * split; ++r)
    good &= tc::ld_cluster_s32(tc::map_rank(tc::smem_u32(&ctl->bad), (uint32_t)r)) == 0;
  if (good) {
    const int nv = min(nc, nj - cb * nc);  // valid columns of this block
    const float tn = ctl->tn;
    const int nl = 1 << tile.l, Hx = tile.Hx, Hy = tile.Hy, Hz = tile.Hz;
    const int* __restrict__ map = LV.map;
    const bool ride = half && LV.l2;
    const float scale = ride ? LV.scale2 : LV.scale;
    double* __restrict__ lc = ride ? LV.lc2 : LV.lc;
    // The rows of this CTA's tile, shared out over the split pairs; a warp
    // writes one (row, class) at a time, its lanes along the coefficients, and
    // finds 32 of them at a time, one per lane: 16,000 cycles (biharmonic
    // p = 8).  An element loop over the whole tile, with index divisions per
    // element and the table norm (FP64) in every thread, took 62,000, 13% of a
    // CTA; converting to double with integer operations took 20,000.
    const int rows = gather ? grows : tile.n;
    const int n0 = rows * sp / split, nr = rows * (sp + 1) / split - n0;
    const uint32_t stg = tc::smem_u32(sm);
    uint32_t part[kMaxSplit];
#pragma unroll
    for (int q = 0; q < kMaxSplit; ++q)
      part[q] = q < split ? tc::map_rank(stg, (uint32_t)(2 * q + half)) : 0u;
    constexpr int kPer = kMaxN / 32;  // coefficients per lane (nc <= 256)
    float f[kPer];                    // F16X3: S_i and the table norm
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const int i = lane + 32 * j;
      f[j] = F::kScaled && i < nv ? prm.fact_f[cb * nc + i] * tn : 1.f;
    }
    const int tot = nr * ncls;  // ncls is a power of two
    const int cshift = __ffs(ncls) - 1;
    const int end = tot * (warp + 1) / kEpiWarps;
    for (int r0 = tot * warp / kEpiWarps; r0 < end; r0 += 32) {
      int64_t mine = -1;  // box of (row, class) r0 + lane
      if (r0 + lane < end) {
        const int n = n0 + ((r0 + lane) >> cshift);
        const int pi = pi0 + ((r0 + lane) & (ncls - 1));
        if (gather) {  // row n: entry gstart + n of the class list
          mine = map[(size_t)pi * Hz * Hy * Hx + LV.tlist[gstart + n]];
        } else {
          const int x = tile.X0 + n % tile.BX, y = tile.Y0 + n / tile.BX % tile.BY,
                    z = tile.Z0 + n / (tile.BX * tile.BY);
          if (x < Hx && y < Hy && z < Hz)
            mine = map ? (int64_t)map[(((size_t)pi * Hz + z) * Hy + y) * Hx + x]
                       : ((int64_t)(2 * z + (pi >> 2)) * nl + (2 * y + ((pi >> 1) & 1))) * nl +
                             (2 * x + (pi & 1));
        }
      }
      const int cnt = min(32, end - r0);
      for (int q = 0; q < cnt; ++q) {
        const int64_t t = __shfl_sync(0xffffffffu, mine, q);
        if (t < 0) continue;
        const int r = r0 + q;
        const int at = (n0 + (r >> cshift)) * (nmma + 1) + (r & (ncls - 1)) * nc + lane;
        double* __restrict__ dst = lc + t * nj + cb * nc + lane;
        float v[kPer];
        if (split == 1) {
#pragma unroll
          for (int j = 0; j < kPer; ++j)
            if (lane + 32 * j < nv) v[j] = reinterpret_cast<const float*>(sm)[at + 32 * j];
        } else {  // all loads of a row in flight, then the sums in rank order
          float w[kMaxSplit][kPer];
#pragma unroll
          for (int p = 0; p < kMaxSplit; ++p)
#pragma unroll
            for (int j = 0; j < kPer; ++j)
              w[p][j] = p < split && lane + 32 * j < nv
                            ? tc::ld_cluster_f32(part[p] + 4u * (uint32_t)(at + 32 * j))
                            : 0.f;
#pragma unroll
          for (int j = 0; j < kPer; ++j) v[j] = ((w[0][j] + w[1][j]) + w[2][j]) + w[3][j];
        }
#pragma unroll
        for (int j = 0; j < kPer; ++j)
          if (lane + 32 * j < nv) {
            // every coefficient is written by one CTA, before anything adds to it
            dst[32 * j] = (double)((F::kScaled ? v[j] * f[j] : v[j]) * scale);
          }
      }
    }
  }
  __syncwarp();
  cta_sync<kThreads>();
  tc::cluster_sync();  // no CTA leaves while another reads its sums or frees the pair's TMEM
  if (warp == 0) tc::tmem_dealloc_pair(tmem, kTmemCols);
}

// ---- host side: tensor maps ---------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

bool make_map(CUtensorMap* m, void* base, int rank, const cuuint64_t* dims,
              const cuuint64_t* strides, const cuuint32_t* box, CUtensorMapDataType dt) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint32_t es[5] = {1, 1, 1, 1, 1};
  return fn(m, dt, (cuuint32_t)rank, base, dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

// Target tile of a parent grid Hx x Hy x Hz: up to 8 x 4 x 4 = 128 parents,
// x fastest.
void tile_shape(int Hx, int Hy, int Hz, TcLevel* v) {
  v->BX = std::min(8, Hx);
  v->BZ = std::min(4, Hz);
  v->BY = std::min(Hy, kBM / (v->BX * v->BZ));
  v->ntx = (Hx + v->BX - 1) / v->BX;
  v->nty = (Hy + v->BY - 1) / v->BY;
  v->ntiles = v->ntx * v->nty * ((Hz + v->BZ - 1) / v->BZ);
}

// the MMA's N and each CTA's half of B for `ncls` stacked classes (N a
// multiple of 32: with one class the rows past nc are the next matrix's, and
// their columns are not read), and the stage ring they allow
template <typename F, int NPASS>
bool set_columns(TcParams* prm, int ncls) {
  using C = Cfg<NPASS>;
  prm->ncls = ncls;
  prm->nmma = ncls == 1 ? (prm->nc + 31) / 32 * 32 : ncls * prm->nc;
  prm->hb_n = ncls == 1 ? 1 : ncls / 2;
  prm->hb_rows = ncls == 1 ? prm->nmma / 2 : prm->nc;
  prm->stage_bytes = C::stage_bytes(prm->nmma / 2);
  prm->nstages = std::min(kMaxStages, (kSmemCap - 1024 - kTailBytes) / prm->stage_bytes);
  // the staging of the sums reuses the stages
  return prm->nstages >= 3 && prm->nmma <= kMaxN &&
         kBM * (prm->nmma + 1) * (int)sizeof(float) <= prm->nstages * prm->stage_bytes;
}

// Pairs per cluster (TcParams::split) for a launch of `pairs` working pairs: a
// pair walks 189 to 216 combinations at 1-2 us, with a start and an end worth
// about ten more, and clusters of 2, 4, 6 and 8 CTAs fit the 152 SMs
// kClusters[split] times (cudaOccupancyMaxActiveClusters).
constexpr int kClusters[kMaxSplit + 1] = {0, 76, 36, 23, 15};
int choose_split(int64_t pairs) {
  int best = 1;
  double cost = 1e30;
  for (int s = 1; s <= kMaxSplit; ++s) {
    const double c = (double)((pairs + kClusters[s] - 1) / kClusters[s]) * (200.0 / s + 10.0);
    if (c < 0.97 * cost) {
      cost = c;
      best = s;
    }
  }
  return best;
}

// the launch parameters that do not depend on the level
template <typename F, int NPASS>
bool common_params(const fmm_plan_s* P, const Workspace& ws, TcParams* prm) {
  using C = Cfg<NPASS>;
  const TcShape sh = tc_shape(P->pd.nj, P->desc.precision);
  std::memset(prm, 0, sizeof(*prm));
  prm->nj = P->pd.nj;
  const int row = C::kRowBytes / (int)sizeof(typename F::T);  // elements per K chunk
  if (sh.row_bytes != C::kRowBytes || ws.tc_jp != sh.jp || ws.tc_mp != sh.npt) return false;
  prm->jchunks = ws.tc_jp / row;
  const int kstep = 32 / (int)sizeof(typename F::T);  // elements of K per MMA
  const KTail kt = k_tail(P->pd.nj, row, C::kHalves);
  prm->packed = kt.t > 0;
  const int kelems = kt.t > 0 ? kt.k0 + 3 * kt.t : P->pd.nj;  // elements of a hi row in use
  prm->ksteps_last = (kelems + kstep - 1) / kstep - (prm->jchunks - 1) * C::kKSteps;
  prm->nc = sh.nc;
  prm->npt = sh.npt;
  prm->wait_cycles = P->tc_wait_cycles > 0 ? P->tc_wait_cycles : tc::kWaitCycles;
  prm->err = &ws.geom->flag;
  return set_columns<F, NPASS>(prm, sh.ncls) && prm->ksteps_last >= 1 &&
         prm->ksteps_last <= C::kKSteps;
}

template <typename F, int NPASS>
size_t smem_bytes(const TcParams& prm) {
  return 1024 + (size_t)prm.nstages * prm.stage_bytes + kTailBytes;
}

// offset matrices A_h (hi and lo) from the derivative tables
template <typename F, int NPASS>
void build_tables(const fmm_plan_s* P, const Workspace& ws, cudaStream_t st, int tlev) {
  using T = typename F::T;
  const PlanDev& pd = P->pd;
  T* thi0 = static_cast<T*>(ws.tc_tmat[0]);
  T* tlo = NPASS == 3 ? static_cast<T*>(ws.tc_tmat[1]) : nullptr;
  const size_t sm = tmat_smem<F>(pd, ws.tc_jp);
  if (sm > 48 * 1024)
    cudaFuncSetAttribute(k_build_tmat<F>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  const KTail kt = k_tail(pd.nj, Cfg<NPASS>::kRowBytes / (int)sizeof(T), Cfg<NPASS>::kHalves);
  k_build_tmat<F><<<dim3(64, tlev, kTmatSplit), 256, sm, st>>>(pd, ws.geom, ws.htab, ws.tc_mp,
                                                               ws.tc_jp, kt, thi0, tlo);
}

// tensor maps of the offset matrices of table level ti
template <typename F, int NPASS>
bool offset_maps(const Workspace& ws, int ti, const TcParams& prm, TcLevel* v) {
  using C = Cfg<NPASS>;
  using T = typename F::T;
  const size_t esz = sizeof(T);
  const CUtensorMapDataType dt = F::kMapType;
  const int JP = ws.tc_jp, NPT = ws.tc_mp, row = C::kRowBytes / (int)esz;
  const size_t per = (size_t)343 * NPT * JP;
  cuuint64_t dA[2] = {(cuuint64_t)JP, (cuuint64_t)343 * NPT};
  cuuint64_t sA[1] = {(cuuint64_t)JP * esz};
  cuuint32_t bA[2] = {(cuuint32_t)row, (cuuint32_t)prm.hb_rows};
  T* thi = static_cast<T*>(ws.tc_tmat[0]) + (size_t)ti * per;
  if (!make_map(&v->H, thi, 2, dA, sA, bA, dt)) return false;
  v->Hlo = v->H;
  if (NPASS == 3) {
    T* tlo = static_cast<T*>(ws.tc_tmat[1]) + (size_t)ti * per;
    if (!make_map(&v->Hlo, tlo, 2, dA, sA, bA, dt)) return false;
  }
  return true;
}

// tensor map of parity-split multipoles Bpar[8][Hz][Hy][Hx][JP], box of
// (bx, by, bz) parents
template <typename F, int NPASS>
bool source_map(CUtensorMap* m, void* base, int JP, int Hx, int Hy, int Hz, int bx, int by,
                int bz) {
  using C = Cfg<NPASS>;
  const size_t esz = sizeof(typename F::T);
  const CUtensorMapDataType dt = F::kMapType;
  const int row = C::kRowBytes / (int)esz;
  cuuint64_t dB[5] = {(cuuint64_t)JP, (cuuint64_t)Hx, (cuuint64_t)Hy, (cuuint64_t)Hz, 8};
  cuuint64_t sB[4] = {(cuuint64_t)JP * esz, (cuuint64_t)JP * esz * Hx,
                      (cuuint64_t)JP * esz * Hx * Hy, (cuuint64_t)JP * esz * Hx * Hy * Hz};
  cuuint32_t bB[5] = {(cuuint32_t)row, (cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bz, 1};
  return make_map(m, base, 5, dB, sB, bB, dt);
}

template <typename F, int NPASS, bool SHORTW, int NCOL, bool ADAPT>
cudaError_t launch_variant(const TcParams& prm, dim3 grid, size_t sm, cudaStream_t st) {
  const auto kern = k_m2l_tc<F, NPASS, SHORTW, NCOL, ADAPT>;
  // per call: the attribute belongs to the current device's context
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(ADAPT ? kTcThreadsA : kTcThreads);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 2 * prm.split;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, prm);
}

template <typename F, int NPASS, bool ADAPT>
cudaError_t launch_contraction(const fmm_plan_s* P, const TcParams& prm, int npairs,
                               cudaStream_t st, bool timed) {
  const size_t sm = smem_bytes<F, NPASS>(prm);
  const TcShape sh = tc_shape(P->pd.nj, P->desc.precision);
  const dim3 grid((unsigned)(2 * prm.split) * npairs, sh.nchunk);
  const bool small = prm.nmma / kColGroups <= kColsSmall;
  if (timed) mark_contraction(P, 0, st);
  cudaError_t e;
  if (prm.wait_cycles < tc::kWaitCycles)  // a test's shortened waits
    e = small ? launch_variant<F, NPASS, true, kColsSmall, ADAPT>(prm, grid, sm, st)
              : launch_variant<F, NPASS, true, kColsLarge, ADAPT>(prm, grid, sm, st);
  else
    e = small ? launch_variant<F, NPASS, false, kColsSmall, ADAPT>(prm, grid, sm, st)
              : launch_variant<F, NPASS, false, kColsLarge, ADAPT>(prm, grid, sm, st);
  if (timed) mark_contraction(P, 1, st);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename F, int NPASS>
cudaError_t run_all_levels(const fmm_plan_s* P, const Workspace& ws, cudaStream_t st,
                           bool tables_ready) {
  const PlanDev& pd = P->pd;
  const int L = P->desc.levels;
  const int nj = pd.nj, JP = ws.tc_jp;
  const bool shared_t = kernel_homogeneous(pd.kernel);  // G(s h) = s^deg G(h)
  const int tlev = shared_t ? 1 : (L - 1);
  using T = typename F::T;
  T* bhi0 = static_cast<T*>(ws.tc_bpar[0]);
  T* blo = NPASS == 3 ? static_cast<T*>(ws.tc_bpar[1]) : nullptr;
  LevOff lo;
  for (int l = 0; l <= FMM_MAX_LEVELS; ++l) lo.o[l] = l <= L + 1 ? ws.lev_off[l] : 0;
  const KTail kt = k_tail(nj, Cfg<NPASS>::kRowBytes / (int)sizeof(T), Cfg<NPASS>::kHalves);
  if (F::kScaled)
    k_pack_beta_scaled<F><<<dim3(152 * 4, L - 1), 256, 0, st>>>(ws.mp, lo, nj, JP, kt, pd.fact_f,
                                                                bhi0, blo, ws.tc_bscale);
  else
    k_pack_beta<F><<<dim3(152 * 4, L - 1), 256, 0, st>>>(ws.mp, lo, nj, JP, kt, bhi0, blo);
  if (!tables_ready) build_tables<F, NPASS>(P, ws, st, tlev);
  TcParams prm;
  if (!common_params<F, NPASS>(P, ws, &prm)) return cudaErrorInvalidValue;
  prm.geom = ws.geom;
  prm.kernel = pd.kernel;
  prm.tlev_fixed = shared_t ? 2 : 0;  // shared tables are level 2's
  prm.fact_f = pd.fact_f;
  const int ngrp = 8 / prm.ncls;
  int nb = 0;  // pairs
  // largest level first: its tiles start earliest; with shared offset
  // matrices level 2 rides along in level 3's CTAs
  const int lmin = (shared_t && L >= 3) ? 3 : 2;
  for (int l = L; l >= lmin; --l) {
    TcLevel& v = prm.lev[prm.nlev++];
    const int nl = 1 << l, H = nl >> 1;
    v.l = l;
    v.l2 = 0;
    tile_shape(H, H, H, &v);
    v.first_pair = nb;
    nb += (v.ntiles + 1) / 2 * ngrp;
    v.lc = ws.lc + ws.lev_off[l] * nj;
    v.map = nullptr;
    v.bscale = F::kScaled ? ws.tc_bscale + ws.lev_off[l] : nullptr;
    v.bscale2 = nullptr;
    v.Hx = v.Hy = v.Hz = H;
    v.scale = 1.0f;
    if (shared_t) {  // Ht_l = Ht_2 * (s_2/s_l)^{-deg}: deg -1 (Laplace), +1 (biharmonic)
      const int k = l - 2;
      v.scale = pd.kernel == FMM_KERNEL_LAPLACE ? std::ldexp(1.0f, k) : std::ldexp(1.0f, -k);
    }
    if (!offset_maps<F, NPASS>(ws, shared_t ? 0 : l - 2, prm, &v)) return cudaErrorInvalidValue;
    if (!source_map<F, NPASS>(&v.S, bhi0 + ws.lev_off[l] * JP, JP, H, H, H, v.BX, v.BY, v.BZ))
      return cudaErrorInvalidValue;
    v.Slo = v.S;
    if (NPASS == 3 &&
        !source_map<F, NPASS>(&v.Slo, blo + ws.lev_off[l] * JP, JP, H, H, H, v.BX, v.BY, v.BZ))
      return cudaErrorInvalidValue;
    if (l == 3 && lmin == 3) {  // level 2: 2 x 2 x 2 parents, beside level 3's one tile
      v.l2 = 2;
      v.lc2 = ws.lc + ws.lev_off[2] * nj;
      v.bscale2 = F::kScaled ? ws.tc_bscale + ws.lev_off[2] : nullptr;
      v.scale2 = 1.0f;
      if (!source_map<F, NPASS>(&v.S2, bhi0 + ws.lev_off[2] * JP, JP, 2, 2, 2, 2, 2, 2))
        return cudaErrorInvalidValue;
      v.S2lo = v.S2;
      if (NPASS == 3 &&
          !source_map<F, NPASS>(&v.S2lo, blo + ws.lev_off[2] * JP, JP, 2, 2, 2, 2, 2, 2))
        return cudaErrorInvalidValue;
    }
  }
  prm.split = choose_split((int64_t)nb * tc_shape(nj, P->desc.precision).nchunk);
  return launch_contraction<F, NPASS, false>(P, prm, nb, st, true);
}

// ---- adaptive trees: every level packed into a dense window ----------------
// (the windows come from the tree's per-level coordinate bounds, read with its
// level offsets)

// the level's boxes into Bpar[sigma][Tz][Ty][Tx][JP] (hi and lo) of a window
// with parent origin W and size H, and map[sigma][Tz][Ty][Tx] = box; one warp
// per box (the box's cell found once, the lanes over its coefficients)
template <typename F>
__global__ void __launch_bounds__(256) k_apack(ATree t, int l, const double* __restrict__ mp,
                                               int nj, int JP, const KTail kt, int W0x, int W0y, int W0z, int Hx,
                                               int Hy, int Hz, typename F::T* __restrict__ bhi,
                                               typename F::T* __restrict__ blo,
                                               int* __restrict__ map) {
  const int b0 = t.loff[l], nbl = t.loff[l + 1] - b0;
  const int lane = threadIdx.x & 31;
  const int nw = (int)((gridDim.x * blockDim.x) >> 5);
  for (int bi = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); bi < nbl; bi += nw) {
    const int b = b0 + bi;
    int c[3];
    demorton3(t.key[b], l, c);
    const int sg = (c[0] & 1) | ((c[1] & 1) << 1) | ((c[2] & 1) << 2);
    const size_t cell =
        (((size_t)sg * Hz + ((c[2] >> 1) - W0z)) * Hy + ((c[1] >> 1) - W0y)) * Hx + ((c[0] >> 1) - W0x);
    const double* src = mp + (size_t)b * nj;
    for (int q = lane; q < JP; q += 32) {
      int part;
      const int qs = row_elem(kt, nj, q, &part);
      const float v = qs >= 0 ? (float)src[qs] : 0.f;
      typename F::T hi, lo;
      F::split(v, hi, lo);
      bhi[cell * JP + q] = part == 2 ? lo : hi;
      if (blo) blo[cell * JP + q] = lo;
    }
    if (lane == 0) map[cell] = t.t1[b] > t.t0[b] ? b : -1;  // only boxes with targets get locals
  }
}

// The target cells of level l (boxes holding targets, parent cell in the
// window with parent origin W and size H) grouped by class: toff[u] is where
// class u starts in tlist, toff[8] the total; inside a class the cells keep
// the boxes' Morton order.  Two passes over blocks of 1,024 boxes: each block's
// class counts (cnt, one row of 8 per block), then, with the counts of the
// blocks before it and of the classes before each class, the positions by warp
// ballots.  (One block of 1,024 threads walking the level took 583 us for the
// 168,000 boxes of level 6 of the 2M-point Plummer tree.)
struct ListWindow {
  int l, W0x, W0y, W0z, Hx, Hy;
};
__device__ __forceinline__ int target_class(const ATree& t, const ListWindow& w, int i, int n,
                                            int* cell) {
  const int b = t.loff[w.l] + i;
  if (i >= n || t.t1[b] == t.t0[b]) return -1;
  int c[3];
  demorton3(t.key[b], w.l, c);
  *cell = (((c[2] >> 1) - w.W0z) * w.Hy + ((c[1] >> 1) - w.W0y)) * w.Hx + ((c[0] >> 1) - w.W0x);
  return (c[0] & 1) | ((c[1] & 1) << 1) | ((c[2] & 1) << 2);
}
__global__ void __launch_bounds__(kListBoxes) k_alist_count(ATree t, ListWindow w,
                                                      int* __restrict__ cnt) {
  __shared__ int total[8];
  if (threadIdx.x < 8) total[threadIdx.x] = 0;
  __syncthreads();
  const int n = t.loff[w.l + 1] - t.loff[w.l];
  int cell;
  const int cls = target_class(t, w, (int)(blockIdx.x * kListBoxes + threadIdx.x), n, &cell);
  for (int u = 0; u < 8; ++u) {
    const unsigned m = __ballot_sync(0xffffffffu, cls == u);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(&total[u], __popc(m));
  }
  __syncthreads();
  if (threadIdx.x < 8) cnt[8 * blockIdx.x + threadIdx.x] = total[threadIdx.x];
}
__global__ void __launch_bounds__(kListBoxes) k_alist(ATree t, ListWindow w,
                                                const int* __restrict__ cnt,
                                                int* __restrict__ tlist, int* __restrict__ toff) {
  __shared__ int wcnt[32][8], base[8], sum[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = t.loff[w.l + 1] - t.loff[w.l];
  if (warp < 8) {  // class `warp`: its total, and its count in the blocks before this one
    int all = 0, before = 0;
    for (int k = lane; k < (int)gridDim.x; k += 32) {
      const int c = cnt[8 * k + warp];
      all += c;
      before += k < (int)blockIdx.x ? c : 0;
    }
    all = __reduce_add_sync(0xffffffffu, all);
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 0) {
      sum[warp] = all;
      base[warp] = before;
    }
  }
  int cell = 0;
  const int cls = target_class(t, w, (int)(blockIdx.x * kListBoxes + threadIdx.x), n, &cell);
  unsigned mine = 0;
  for (int u = 0; u < 8; ++u) {
    const unsigned m = __ballot_sync(0xffffffffu, cls == u);
    if (lane == 0) wcnt[warp][u] = __popc(m);
    if (cls == u) mine = m;
  }
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x < 9) {
    int acc = 0;
    for (int u = 0; u < (int)threadIdx.x; ++u) acc += sum[u];
    toff[threadIdx.x] = acc;
  }
  if (cls >= 0) {
    int pos = base[cls] + __popc(mine & ((1u << lane) - 1u));
    for (int u = 0; u < cls; ++u) pos += sum[u];
    for (int q = 0; q < warp; ++q) pos += wcnt[q][cls];
    tlist[pos] = cell;
  }
}

template <typename F, int NPASS>
cudaError_t run_adaptive(const fmm_plan_s* P, const Workspace& ws, const ATree& t,
                         cudaStream_t st, int* nl, unsigned* done) {
  using T = typename F::T;
  const PlanDev& pd = P->pd;
  const int nj = pd.nj, JP = ws.tc_jp;
  const bool shared_t = kernel_homogeneous(pd.kernel);  // G(s h) = s^deg G(h)
  const size_t esz = sizeof(T);
  // coordinate bounds of every level, read with the tree's level offsets
  const int* bnd = P->abnd;
  TcParams prm;
  if (!common_params<F, NPASS>(P, ws, &prm)) return cudaErrorInvalidValue;
  // gathered rows belong to one class: no stacked classes
  if (!set_columns<F, NPASS>(&prm, 1)) return cudaErrorInvalidValue;
  const KTail kt = k_tail(nj, Cfg<NPASS>::kRowBytes / (int)esz, Cfg<NPASS>::kHalves);
  const int nchunk = tc_shape(nj, P->desc.precision).nchunk;
  int64_t working = 0;  // pairs of the launch that have work, about
  const int ngrp = 8;
  int nb = 0;  // pairs
  char* arena = static_cast<char*>(ws.tc_arena);
  size_t used = 0;
  const size_t cell_bytes = (size_t)JP * esz;
  for (int l = t.maxlev; l >= 2; --l) {  // largest (finest) level first
    if (bnd[6 * l + 3] < 0) continue;    // no box at this level
    int W0[3], H[3];
    for (int k = 0; k < 3; ++k) {
      W0[k] = bnd[6 * l + k] >> 1;
      H[k] = (bnd[6 * l + 3 + k] >> 1) - W0[k] + 1;
    }
    const size_t cells = (size_t)8 * H[0] * H[1] * H[2];
    const unsigned nbl = (unsigned)(t.loff[l + 1] - t.loff[l]);
    // a window less than 4/5 full is contracted over its target cells alone
    // (the source rows gathered); a fuller one in tiles of the window.  On the
    // 2M-point Plummer tree (BF16x3, p = 12) a combination of 256 rows takes
    // 3,190 cycles in tiles and 3,480 to 4,050 gathered (levels 6 to 8, 64%, 43%
    // and 39% full); gathering level 6 too took the M2L phase from 7.6 to 6.3 ms.
    const bool gather = 1.25 * (double)nbl < (double)cells;
    auto a256 = [](size_t x) { return (x + 255) / 256 * 256; };
    const size_t rows = cells + (gather ? 1 : 0);  // gathered: a zero row at the end
    const size_t need = a256(rows * cell_bytes) * (NPASS == 3 ? 2 : 1) +
                        a256(cells * sizeof(int)) +
                        (gather ? a256((size_t)nbl * sizeof(int)) + 256 : 0);
    if (need > ws.tc_arena_bytes) continue;  // a window larger than the arena: CUDA cores
    if (used + need > ws.tc_arena_bytes || prm.nlev == kTcMaxLevels) {
      // contract the levels packed so far, then pack the next ones into the
      // same arena (the stream orders the packing after that launch)
      prm.split = choose_split(working * nchunk);
      const cudaError_t e = launch_contraction<F, NPASS, true>(P, prm, nb, st, false);
      ++*nl;
      if (e != cudaSuccess) return e;
      prm.nlev = 0;
      nb = 0;
      working = 0;
      used = 0;
    }
    char* at = arena + used;
    T* bhi = reinterpret_cast<T*>(at);
    at += a256(rows * cell_bytes);
    T* blo = nullptr;
    if (NPASS == 3) {
      blo = reinterpret_cast<T*>(at);
      at += a256(rows * cell_bytes);
    }
    int* map = reinterpret_cast<int*>(at);
    at += a256(cells * sizeof(int));
    int* tlist = gather ? reinterpret_cast<int*>(at) : nullptr;
    int* toff = gather ? reinterpret_cast<int*>(at + a256((size_t)nbl * sizeof(int))) : nullptr;
    used += need;
    cudaMemsetAsync(bhi, 0, rows * cell_bytes, st);
    if (blo) cudaMemsetAsync(blo, 0, rows * cell_bytes, st);
    cudaMemsetAsync(map, 0xff, cells * sizeof(int), st);
    k_apack<F><<<std::min<unsigned>((nbl + 7) / 8, 152 * 16), 256, 0, st>>>(
        t, l, ws.mp, nj, JP, kt, W0[0], W0[1], W0[2], H[0], H[1], H[2], bhi, blo, map);
    ++*nl;
    if (gather) {
      const ListWindow lw{l, W0[0], W0[1], W0[2], H[0], H[1]};
      // the counts go to the scratch of the tree build's tickets
      if (alist_counts(nbl) > ws.ascan_n) return cudaErrorInvalidValue;
      const unsigned nblk = (nbl + kListBoxes - 1) / kListBoxes;
      k_alist_count<<<nblk, kListBoxes, 0, st>>>(t, lw, ws.ascan);
      k_alist<<<nblk, kListBoxes, 0, st>>>(t, lw, ws.ascan, tlist, toff);
      *nl += 2;
    }
    TcLevel& v = prm.lev[prm.nlev++];
    v.l = l;
    v.l2 = 0;
    v.Hx = H[0];
    v.Hy = H[1];
    v.Hz = H[2];
    v.gather = gather ? 1 : 0;
    v.tlist = tlist;
    v.toff = toff;
    v.zero_row = (int)cells;
    v.first_pair = nb;
    if (gather) {  // 256 list entries per pair, the classes interleaved; a class holds at
                   // most one cell per parent of the window
      v.BX = 8;
      v.BY = 4;
      v.BZ = 4;
      v.ntx = v.nty = v.ntiles = 1;
      const size_t per_cls = std::min<size_t>(nbl, cells / 8);
      nb += 8 * (int)((per_cls + 2 * kBM - 1) / (2 * kBM));
      working += 8 * (int64_t)((nbl / 8 + 2 * kBM - 1) / (2 * kBM));
    } else {
      tile_shape(H[0], H[1], H[2], &v);
      nb += (v.ntiles + 1) / 2 * ngrp;
      working += (v.ntiles + 1) / 2 * ngrp;
    }
    v.lc = ws.lc;
    v.map = map;
    v.scale = 1.0f;
    if (shared_t) {
      const int k = l - 2;
      v.scale = pd.kernel == FMM_KERNEL_LAPLACE ? std::ldexp(1.0f, k) : std::ldexp(1.0f, -k);
    }
    if (!offset_maps<F, NPASS>(ws, shared_t ? 0 : l - 2, prm, &v)) return cudaErrorInvalidValue;
    v.ghi = reinterpret_cast<const char*>(bhi);
    v.glo = reinterpret_cast<const char*>(NPASS == 3 ? blo : bhi);
    if (!gather) {
      if (!source_map<F, NPASS>(&v.S, bhi, JP, H[0], H[1], H[2], v.BX, v.BY, v.BZ))
        return cudaErrorInvalidValue;
      v.Slo = v.S;
      if (NPASS == 3 &&
          !source_map<F, NPASS>(&v.Slo, blo, JP, H[0], H[1], H[2], v.BX, v.BY, v.BZ))
        return cudaErrorInvalidValue;
    }
    *done |= 1u << l;
  }
  if (prm.nlev == 0) return cudaGetLastError();
  prm.split = choose_split(working * nchunk);
  const cudaError_t r = launch_contraction<F, NPASS, true>(P, prm, nb, st, false);
  ++*nl;
  return r;
}

}  // namespace

cudaError_t launch_m2l_tc(const fmm_plan_s* P, const Workspace& ws, cudaStream_t st, int* nl,
                          bool tables_ready) {
  const int L = P->desc.levels;
  if (P->pd.d != 3) {
    cudaMemsetAsync(ws.lc, 0, sizeof(double) * (size_t)ws.lev_off[L + 1] * P->pd.nj, st);
    return launch_m2l_simt_levels(P, ws, 2, L, st, nl);
  }
  const int prec = P->desc.precision;
  const cudaError_t e =
      prec == FMM_PREC_F16X3    ? run_all_levels<FmtF16, 3>(P, ws, st, tables_ready)
      : prec == FMM_PREC_BF16X3 ? run_all_levels<FmtBF16, 3>(P, ws, st, tables_ready)
      : prec == FMM_PREC_TF32X3 ? run_all_levels<FmtTF32, 3>(P, ws, st, tables_ready)
                                : run_all_levels<FmtTF32, 1>(P, ws, st, tables_ready);
  *nl += tables_ready ? 2 : 3;
  return e;
}

// the offset matrices alone (3D tree of levels 0..maxlev, tensor-core precisions), so
// that they can be built on another stream ahead of the contraction
cudaError_t launch_m2l_tc_tables(const fmm_plan_s* P, const Workspace& ws, int maxlev,
                                 cudaStream_t st, int* nl) {
  const int prec = P->desc.precision;
  const int tlev = kernel_homogeneous(P->pd.kernel) ? 1 : maxlev - 1;
  if (prec == FMM_PREC_F16X3) build_tables<FmtF16, 3>(P, ws, st, tlev);
  else if (prec == FMM_PREC_BF16X3) build_tables<FmtBF16, 3>(P, ws, st, tlev);
  else if (prec == FMM_PREC_TF32X3) build_tables<FmtTF32, 3>(P, ws, st, tlev);
  else build_tables<FmtTF32, 1>(P, ws, st, tlev);
  ++*nl;
  return cudaGetLastError();
}

// (launch_m2l_tc_tables has been ordered before)
cudaError_t launch_adaptive_m2l_tc(const fmm_plan_s* P, const Workspace& ws, const ATree& t,
                                   cudaStream_t st, int* nl, unsigned* done) {
  *done = 0;
  if (t.maxlev < 2) return cudaGetLastError();
  const int prec = P->desc.precision;
  return prec == FMM_PREC_BF16X3   ? run_adaptive<FmtBF16, 3>(P, ws, t, st, nl, done)
         : prec == FMM_PREC_TF32X3 ? run_adaptive<FmtTF32, 3>(P, ws, t, st, nl, done)
                                   : run_adaptive<FmtTF32, 1>(P, ws, t, st, nl, done);
}
