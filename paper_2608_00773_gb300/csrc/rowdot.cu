// Split-precision density (Eqs. 39-40) and adjoint of the integration on the
// tcgen05 tensor cores.
//
// Both are row-dot contractions over the batch's active functions:
//   density   n_p     = sum_ij P_ij Phi_pi Phi_pj
//   adjoint   dL/dv_p = w_p [ sum_ij G^V_ij Phi_i Phi_j + sum_{Q=X,Y,Z} sum_ij G^W_ij Q_i Q_j
//                             + sum_ij (G^x_ij - G^x_ji) Y_i Z_j + (cyclic) ](p)
// (the cross product is antisymmetric in i, j, so only G - G^T of the SO
// matrices enters).  For P, G^V and G^W only the symmetric part enters, so the
// sum runs over i <= j with G_ij + G_ji off the diagonal: half the products.
// Each is U = F G' (rows = points, K = functions i, columns = functions j)
// dotted with R in the epilogue, one point per tensor-memory lane; the products
// of one adjoint are (F, G', R) = (Phi, V, Phi), (Q, W, Q), (Y, x, Z), (Z, y, X),
// (X, z, Y).
//
// Each U is computed from six BF16 slices of F (an exponent per point and
// quantity) and of G' (an exponent per column and matrix) in six FP32
// accumulators, one per level s + t (see split.cu): levels 0-2 are exact integer
// sums for K <= 204 terms (kFine; here at most 112), levels 3-5 are rounded 2^-24
// below.
//
// G' does not depend on the points, so a pre-pass slices every batch's G' once
// into BF16 digit tiles laid out exactly as the MMA reads them (per matrix,
// 32-function j-tile and 16-function i-chunk: six tiles of up to 32 rows); the
// main kernel streams them with bulk copies.
#include <algorithm>

#include "internal.h"
#include "tc.cuh"

namespace q4c {
namespace rowdot {
using namespace tc;

constexpr int kPts = 128;                      // points per item (MMA rows, tensor-memory lanes)
constexpr int kTileJ = 32;                     // functions j per tile
constexpr int kKc = 16;                        // functions i per chunk (one K = 16 MMA step)
constexpr int kSBO = (kKc / 8) * 128;          // 256 B between 8-row groups
constexpr int kDigA = kPts * kKc * 2;          // one digit tile of F, 4 KB
constexpr int kSlot = kSlices * kDigA;         // one chunk of F, 24 KB
constexpr int kSlots = 7;                      // resident chunks
constexpr int kBlockB = kSlices * kTileJ * kRowBytes;  // one step's G' digits, up to 6 KB
constexpr int kRingB = 4;                      // G' blocks in flight per accumulator set
// 16 warps, so that the epilogue has 128 registers a thread
constexpr int kSlicers = 128;                  // warps 0-3 slice F
constexpr int kEpiWarp0 = 4;                   // warps 4-11 drain tensor memory (two groups of four)
constexpr int kEpiThreads = 256;
constexpr int kMmaWarp = 12;   // warps 12 and 13 issue the MMAs, one per accumulator set; 12 owns tensor memory
constexpr int kProdWarp = 14;  // warps 14 and 15 stream the G' blocks, one per accumulator set
constexpr int kThreads = 16 * 32;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kSetCols = 256;  // two accumulator sets of six levels of up to 32 columns
constexpr int kMaxNb = 4096;
// The digits resolve 2^-2 finer than tc::slice6x2 does against the exponent
// itself: with |d_0| <= 256 (exact in BF16) a term of the exact levels is at most
// 2 * 256 * 128 + 128^2 units, so that they hold 204 terms below 2^24, and the symmetric matrices'
// doubled coefficients are resolved as finely as their two halves were (error of
// the 64-atom density against FP64: 1.5e-13 before, 2.7e-13 at the coarser
// digits, 4.7e-14 with these).
constexpr int kFine = 2;

// Shared memory: the F slots, a ring of G' blocks per accumulator set (KS blocks
// per stage: the stage shape the tuner chooses), the points' partial sums and
// the barriers.
template <int KS>
struct Layout {
  static constexpr int kStages = kRingB / KS;  // of one ring
  static constexpr int kStage = KS * kBlockB;
  static constexpr int kSmemRing = kSlots * kSlot;
  static constexpr int kSmemY = kSmemRing + 2 * kStages * kStage;  // [2][128] double partials per point
  static constexpr int kSmemBar = kSmemY + 2 * kPts * 8;
  // slot full/empty, stage full/empty of both rings, accfull[2], accempty[2], drain[2]
  static constexpr int kNumBars = 2 * kSlots + 4 * kStages + 6;
  static constexpr int kSmemTotal = kSmemBar + kNumBars * 8 + 16;
  static_assert(kSmemTotal <= 232448, "shared memory per CTA");
};

// ------------------------------------------------------------ preparation
struct Mats {
  const double* m[5];
};

// One CTA per pattern block q (A, B, T) (grid-stride), every present matrix: the
// FP32-pair copies (hi + lo within 2^-48 relative) of what a pair i <= j of a
// batch takes from the block, G + G^T for V and W (G itself on the diagonal of
// a block that is its own partner) and G - G^T for the SO matrices, formed in
// FP64, G^T read from the partner block (B, A, -T) through shared memory where
// both sides have at most 64 functions, else straight from memory; and at
// cm_off[q] an FP32 bound of each of its nf_B columns, cm[m] for matrix m.
__global__ void __launch_bounds__(128) k_prepare_blocks(DevBasis B, DevGrid G, Mats M, int64_t n_blocks,
                                                       const int* __restrict__ blk_row,
                                                       const int* __restrict__ blk_col,
                                                       const int64_t* __restrict__ blk_off,
                                                       const int* __restrict__ blk_T,
                                                       const int64_t* __restrict__ cm_off, float2* __restrict__ out,
                                                       int64_t nnz, float* __restrict__ cm, int64_t cm_total) {
  __shared__ double sT[64 * 65];      // G^T of the block: sT[i * 65 + j] = partner (j, i)
  extern __shared__ unsigned s_cm[];  // [5][nf_B] bits of the column bounds (non-negative floats order as integers)
  for (int64_t q = blockIdx.x; q < n_blocks; q += gridDim.x) {
    const int nfA = __ldg(B.sp_nfn + G.atom_sp[blk_row[q]]), nfB = __ldg(B.sp_nfn + G.atom_sp[blk_col[q]]);
    const int64_t o0 = blk_off[q];
    const int ne = nfA * nfB, qt = blk_T[q];
    const bool tile = qt >= 0 && nfA <= 64 && nfB <= 64;
    __syncthreads();
    for (int j = threadIdx.x; j < 5 * nfB; j += blockDim.x) s_cm[j] = 0u;
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      if (M.m[m] == nullptr) continue;
      const double* X = M.m[m] + o0;
      const double* XT = qt >= 0 ? M.m[m] + blk_off[qt] : nullptr;  // nfB rows x nfA columns
      __syncthreads();
      if (tile) {
        for (int e = threadIdx.x; e < ne; e += blockDim.x) {
          const int r = e / nfA, c = e - r * nfA;
          sT[c * 65 + r] = XT[e];
        }
        __syncthreads();
      }
      float2* o = out + m * nnz + o0;
      for (int e = threadIdx.x; e < ne; e += blockDim.x) {
        const int i = e / nfB, j = e - i * nfB;
        const double xt = tile ? sT[i * 65 + j] : XT ? XT[static_cast<int64_t>(j) * nfA + i] : 0.0;
        const double g = X[e];
        const double x = m >= 2 ? g - xt : (qt == q && i == j) ? g : g + xt;
        const float h = __double2float_rn(x), l = __double2float_rn(x - static_cast<double>(h));
        o[e] = make_float2(h, l);
        atomicMax(&s_cm[m * nfB + j], __float_as_uint(__fadd_ru(fabsf(h), fabsf(l))));
      }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < nfB; j += blockDim.x)
#pragma unroll
      for (int m = 0; m < 5; ++m)
        if (M.m[m]) cm[m * cm_total + cm_off[q] + j] = __uint_as_float(s_cm[m * nfB + j]);
  }
}

__device__ __forceinline__ int fexp(float x) {  // |x| < 2^fexp(x) for x != 0
  return static_cast<int>((__float_as_uint(x) >> 23) & 0xFF) - 126;
}

// width of j-tile jt: its functions rounded up to 16 (the MMA's N
// granularity); its G' digit tiles hold that many rows
__host__ __device__ __forceinline__ int jt_width(int nb, int jt) {
  const int w = nb - jt * kTileJ;
  return ((w < kTileJ ? w : kTileJ) + 15) & ~15;
}

// chunks of i that matrix m has in j-tile jt: all of them, or for V and W those
// up to the tile's last column
__host__ __device__ __forceinline__ int jt_chunks(int m, int n_ic, int jt) {
  const int n = 2 * (jt + 1);
  return m < 2 && n < n_ic ? n : n_ic;
}

// Pre-pass: CTAs (batch, share of the j-tiles), all NM matrices (V alone or the
// five).  Per j-tile the column exponents e_j (|G'_ij| < 2^e_j over the batch's i),
// then the six digits of every G'_ij written as the B operand of the main kernel:
// block (jt, ic) = six tiles of jt_width rows (j) x 16 K (i), 32 bytes a row, in
// the no-swizzle K-major layout, back to back, at (jt * n_ic) * 6 KB + ic * 192 *
// jt_width; padding rows and columns, and for V and W i > j, are 0.
// The column bound is the largest column bound (k_prepare_blocks) of the blocks
// (a, c) of column j's centre c over the batch's active centres a, whose
// functions are exactly the batch's i.
// What bounds it: the stores (12 bytes an element and matrix; 5.5 TB/s with the reads
// on batches of 900 functions).  A warp takes units of 8 j x 8 i (32 words of a tile, an
// element pair each), so a unit's place needs no division and its offsets are read
// once for all matrices.  One matrix a CTA with offsets and divisions of its own:
// 24 molecules 6.8 ms -> 4.0, 64-atom cluster 0.60 -> 0.39, 304-atom slab 12.1 ->
// 10.7.  Forty warps an SM with one unit's ten values in flight each: two units a
// turn 4.4, 0.43 and 12.5 ms at 32 warps, 3.8, 0.38 and 11.6 at 48.
template <int NM>
__global__ void __launch_bounds__(256, 5) k_gslice(DevGrid G, int64_t b0, const float2* __restrict__ prep, int64_t nnz,
                                                unsigned present, const float* __restrict__ cm, int64_t cm_total,
                                                const int* __restrict__ pair_blk, const int64_t* __restrict__ cm_off,
                                                const int64_t* __restrict__ gsl_off, uint32_t* __restrict__ gsl) {
  __shared__ unsigned sMax[NM][kTileJ];  // column bounds per matrix (bits)
  const int64_t b = b0 + blockIdx.x;
  const int64_t f0 = G.bat_fn_ptr[b];
  const int nb = static_cast<int>(G.bat_fn_ptr[b + 1] - f0);
  const int* idx = G.bat_idx + G.bat_idx_ptr[b];
  const int n_jt = (nb + kTileJ - 1) / kTileJ, n_ic = (nb + kKc - 1) / kKc;
  const int na = G.bat_atom_ptr[b + 1] - G.bat_atom_ptr[b];
  const int* pb = pair_blk + G.bat_pair_ptr[b];
  uint32_t* out = gsl + gsl_off[b] / 4;
  const int64_t mstride = static_cast<int64_t>(n_jt) * n_ic * (kBlockB / 4);  // words of one matrix
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  const int r8 = lane >> 2, kp = lane & 3;
  for (int jt = blockIdx.y; jt < n_jt; jt += gridDim.y) {
    __syncthreads();
    if (threadIdx.x < NM * kTileJ) sMax[threadIdx.x / kTileJ][threadIdx.x % kTileJ] = 0u;
    __syncthreads();
    {  // column bounds: eight threads a column over the batch's centres
      const int jl = threadIdx.x >> 3, j = jt * kTileJ + jl;
      if (j < nb) {
        const int info = G.fn_info[f0 + j], c = info >> 16, jj = info & 0xffff;
        float mx[NM] = {};
        for (int a = threadIdx.x & 7; a < na; a += 8) {
          const int q = pb[a * na + c];  // block (a, c): its column jj
          if (q >= 0) {
            const int64_t o = cm_off[q] + jj;
#pragma unroll
            for (int m = 0; m < NM; ++m)
              if (present >> m & 1u) mx[m] = fmaxf(mx[m], __ldg(cm + m * cm_total + o));
          }
        }
#pragma unroll
        for (int m = 0; m < NM; ++m) atomicMax(&sMax[m][jl], __float_as_uint(mx[m]));
      }
    }
    __syncthreads();
    const int w = jt_width(nb, jt), tw = w * 8;  // words of one tile (one per element pair)
    const int sh = w == kTileJ ? 3 : 2;          // log2 of a block's units, w / 4
    const int n_low = jt_chunks(0, n_ic, jt) << sh;  // units that V and W have
    const int units = (present & ~3u) ? n_ic << sh : n_low;
    uint32_t* oj = out + static_cast<int64_t>(jt) * n_ic * (kBlockB / 4);
    // a warp takes kU units at a time and issues all their loads (addresses
    // clamped, conditions the same for the whole warp) before slicing any
    constexpr int kU = NM > 1 ? 1 : 4;
    for (int u0 = warp; u0 < units; u0 += kU * nwarps) {
      int i_[kU], j_[kU], o0[kU], o1[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int un = u0 + u * nwarps, r = un & ((1 << sh) - 1);
        i_[u] = (un >> sh) * kKc + (r & 1) * 8 + kp * 2;
        j_[u] = (r >> 1) * 8 + r8;
        const int j = min(jt * kTileJ + j_[u], nb - 1);
        o0[u] = __ldg(idx + min(i_[u], nb - 1) * nb + j);
        o1[u] = __ldg(idx + min(i_[u] + 1, nb - 1) * nb + j);
      }
      bool ok0[kU], ok1[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const bool jin = jt * kTileJ + j_[u] < nb;
        ok0[u] = jin && i_[u] < nb && o0[u] >= 0;
        ok1[u] = jin && i_[u] + 1 < nb && o1[u] >= 0;
        o0[u] = ok0[u] ? o0[u] : 0;
        o1[u] = ok1[u] ? o1[u] : 0;
      }
      float2 x0[NM][kU], x1[NM][kU];
#pragma unroll
      for (int m = 0; m < NM; ++m)
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          if (!(present >> m & 1u) || u0 + u * nwarps >= (m < 2 ? n_low : units)) continue;
          x0[m][u] = __ldg(prep + m * nnz + o0[u]);
          x1[m][u] = __ldg(prep + m * nnz + o1[u]);
        }
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        if (!(present >> m & 1u)) continue;
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          const int un = u0 + u * nwarps;
          if (un >= (m < 2 ? n_low : units)) break;
          const int j = jt * kTileJ + j_[u];
          const bool a0 = ok0[u] && (m >= 2 || i_[u] <= j), a1 = ok1[u] && (m >= 2 || i_[u] + 1 <= j);
          const float2 y0 = x0[m][u], y1 = x1[m][u];
          const unsigned mb = sMax[m][j_[u]];
          float2 d[kSlices];
          slice6x2(pk2(a0 ? y0.x : 0.f, a1 ? y1.x : 0.f), pk2(a0 ? y0.y : 0.f, a1 ? y1.y : 0.f),
                   magic0((mb ? fexp(__uint_as_float(mb)) : -30000) - kFine), d);
          uint32_t* o = oj + m * mstride + (un >> sh) * (kSlices * tw) + ((un & ((1 << sh) - 1)) << 5) + lane;
#pragma unroll
          for (int t = 0; t < kSlices; ++t) o[t * tw] = bf16x2_exact(d[t]);
        }
      }
    }
  }
}

// ------------------------------------------------------------ the walk
// Work of one item (batch, 128-point tile, j-tiles [jt0, jt1): all of them, or
// a share of a large batch's), the same for every warp role.
//
// Chunks of F digits stay in shared memory while every product that reads them
// runs: an item is a list of segments, a segment fills up to seven slots and
// then runs its groups, and a group (j-tile, R, a run of chunks) is one
// accumulation drained by the epilogue.
// An item has K segments of up to seven chunks, in each one segment per quantity,
// whose groups are single products (the row-dot with R is linear in U, so K
// segments add up in the point's running sum).  Two products that are dotted with
// the same R (W with F = R and an SO matrix) would share an accumulation only at
// the price of one exponent for X, Y and Z of a point: on points along an axis,
// X 2e4 times smaller than Z, the adjoint of SO_z alone then lost 14 bits of F.
struct Item {
  int64_t bp0, scr, gsl, part, plane;
  int pt, np, ldp, nb, n_jt, n_ic;
  int jt0, jt1;  // the item's j-tiles
  int seg_len, nq;  // chunks of a K segment, segments in one
  unsigned qlist;  // quantities of a K segment, two bits each
};

struct Seg {
  int q, c0, c1, n;  // quantity and chunks [c0, c1); n: entries (slots)
};

// the SO matrix that multiplies F = quantity q (X: z, Y: x, Z: y) and the
// quantity it is dotted with
__device__ __forceinline__ int so_matrix(int q) { return q == 1 ? 4 : q + 0; }
__device__ __forceinline__ int so_dot(int q) { return q == 3 ? 1 : q + 1; }

template <int MODE>
__device__ __forceinline__ Item item_of(const RdItem* __restrict__ it, unsigned present) {
  const int4 u = __ldg(reinterpret_cast<const int4*>(it));
  const longlong2 v = __ldg(reinterpret_cast<const longlong2*>(it) + 1), w = __ldg(reinterpret_cast<const longlong2*>(it) + 2);
  Item I;
  I.pt = u.z;
  I.jt0 = u.w & 0xffff;
  I.jt1 = u.w >> 16;
  I.bp0 = v.x;
  I.scr = v.y;
  I.gsl = w.x;
  I.part = w.y;
  I.np = u.x;
  I.nb = u.y;
  I.ldp = (I.np + 7) & ~7;
  I.n_jt = (I.nb + kTileJ - 1) / kTileJ;
  I.n_ic = (I.nb + kKc - 1) / kKc;
  I.plane = static_cast<int64_t>(I.nb) * I.ldp;
  const int n_kseg = max((I.n_ic + kSlots - 1) / kSlots, 1);
  I.seg_len = n_kseg == 1 ? I.n_ic : (I.n_ic + n_kseg - 1) / n_kseg;
  I.qlist = 0;
  I.nq = 0;
  if (MODE == 0 || (present & 1u)) ++I.nq;  // Phi (two zero bits)
  if (MODE == 1) {
#pragma unroll
    for (int q = 1; q < 4; ++q)
      if (present & (2u | 1u << so_matrix(q))) I.qlist |= static_cast<unsigned>(q) << (2 * I.nq++);
  }
  if (I.n_ic == 0) I.nq = 0;
  return I;
}

// segment qi of the K segment that starts at chunk c0
template <int MODE>
__device__ __forceinline__ Seg seg_of(const Item& I, int qi, int c0, unsigned present) {
  const int q = MODE == 0 ? 0 : static_cast<int>((I.qlist >> (2 * qi)) & 3u);
  // a symmetric matrix alone needs the chunks up to the last j-tile's end only
  const bool sym = q == 0 || !(present >> so_matrix(q) & 1u);
  const int c1 = min(sym ? min(I.n_ic, 2 * I.jt1) : I.n_ic, c0 + I.seg_len);
  return {q, c0, c1, max(0, c1 - c0)};
}
// the segment after (qi, c0); false past the item's last one
__device__ __forceinline__ bool next_seg(const Item& I, int& qi, int& c0) {
  if (++qi < I.nq) return true;
  qi = 0;
  c0 += I.seg_len;
  return c0 < I.n_ic;
}

// The groups of one item in order: open() an item, then next() until it
// returns false.
template <int MODE>
struct GroupWalk {
  Item I;
  Seg S;
  unsigned present;
  int ent = 0;          // first entry of the segment in the CTA's sequence
  int qi, c0, part, jt;  // qi = -1: before the item's first segment
  int qr;               // quantity of the dot
  int m, n;             // matrix, chunks (the segment's first n)
  bool last;            // last group of its segment: it reads every chunk
  __device__ __forceinline__ explicit GroupWalk(unsigned pr) : present(pr) { S.n = 0; }
  __device__ __forceinline__ void open(const RdItem* it) {
    I = item_of<MODE>(it, present);
    qi = -1;
    c0 = 0;
  }
  __device__ __forceinline__ bool has(int k) const { return present >> k & 1u; }
  __device__ __forceinline__ bool next() {
    for (;;) {
      if (qi >= 0 && part < 2) {
        ++jt;
        const int mt = S.q ? 1 : 0;  // the symmetric matrix
        const bool so = MODE == 1 && S.q && has(so_matrix(S.q));
        if (jt >= I.jt1) {
          ++part;
          jt = I.jt0 - 1;
          continue;
        }
        if (part == 0) {
          n = min(S.c1, jt_chunks(mt, I.n_ic, jt)) - S.c0;
          if (n <= 0 || !(MODE == 0 || has(mt))) continue;
          m = mt;
          qr = S.q;
          last = !so && jt + 1 == I.jt1;
        } else {
          if (!so) continue;
          m = so_matrix(S.q);
          n = S.n;
          qr = so_dot(S.q);
          last = jt + 1 == I.jt1;
        }
        return true;
      }
      // the next segment
      ent += S.n;
      S.n = 0;
      if (I.nq == 0 || !next_seg(I, qi, c0)) return false;
      S = seg_of<MODE>(I, qi, c0, present);
      part = 0;
      jt = I.jt0 - 1;
    }
  }
};

// The entries (chunks of F) of this CTA's items in order.
template <int MODE>
struct EntryWalk {
  const RdItem* items;
  int n_items;
  unsigned present;
  int n, qi, c0, e;  // item, segment, entry within it: chunk S.c0 + e of quantity S.q
  Item I;
  Seg S;
  __device__ __forceinline__ EntryWalk(const RdItem* it, int ni, unsigned pr)
      : items(it), n_items(ni), present(pr), n(static_cast<int>(blockIdx.x)), e(-1) {
    if (n < n_items) open();
  }
  __device__ __forceinline__ void open() {
    I = item_of<MODE>(items + n, present);
    qi = c0 = 0;
    S.n = 0;
    if (I.nq) S = seg_of<MODE>(I, 0, 0, present);
  }
  // advances to the next entry; false at the end
  __device__ __forceinline__ bool next() {
    if (n >= n_items) return false;
    ++e;
    while (e >= S.n) {
      e = 0;
      if (I.nq && next_seg(I, qi, c0)) {
        S = seg_of<MODE>(I, qi, c0, present);
      } else {
        n += gridDim.x;
        if (n >= n_items) return false;
        open();
      }
    }
    return true;
  }
};

// The 21 slice products of one step (s + t <= 5) as six MMAs: digit tile A_s
// (128 points) times the consecutive digit tiles B_0 .. B_(5-s) (w columns
// each) adds level s + t to columns [(s + t) w, (s + t + 1) w).
__device__ __forceinline__ void mma_row_levels(uint32_t tmem, uint64_t a, uint64_t b, int w, bool first) {
#pragma unroll
  for (int s = 0; s < kSlices; ++s)
    mma_bf16(tmem + s * w, a + s * (kDigA >> 4), b, make_idesc(128, w * (kSlices - s)), (first && s == 0) ? 0u : 1u);
}

// One work item = (batch, 128-point tile).  Warp roles (one persistent CTA per
// SM, items strided over the CTAs):
//   warps 0-3   slice F: thread = point, chunks of 16 functions: reads its raw
//               values straight from the basis tiles one chunk ahead, waits for
//               the slot (slot_empty), stores the six digits of its row, arrives
//               on slot_full;
//   warps 14-15 (one thread each) stream the G' blocks of one accumulator set's
//               groups in order into its ring, KS blocks per bulk copy (g_full
//               counts the bytes), and prefetch the next item's rows into L2;
//   warps 12-13 issue six MMAs per chunk into the group's accumulator set
//               (groups alternate between two sets, a warp each), commit
//               g_empty per stage, slot_empty after a slot's last use (each
//               warp its own) and acc_full after the group;
//   warps 4-11  read the six levels from tensor memory (lane = point, each group
//               of four warps half of the columns; R one group ahead), form U = exact levels by
//               two-sums plus the rounded tail, dot with R in double-float, and
//               write each point's result (of a share, its part) at the end of the item.
// Warps whose points lie past n_p slice and drain nothing.
// Every wait is bounded; a timeout sets the status bit and an abort flag.
//
// What bounds it: a step reads 46 KB of operands from shared memory (six times
// 4 KB of F, 672 rows of 32 B of G'), 360 clocks at 128 B a clock (336 of tensor
// work), and the 6 KB of its G' block arrive there; slicing (once per quantity
// and chunk) and the epilogue (28 FP32 operations per element) share the FP32
// lanes.  Before, 64-point items re-sliced F for every product and 64-column
// tile, and their epilogue ran over two half-level sums of all seven products:
// 89 KB through shared memory a step and 1,360 clocks.
// Adjoint, before -> now: 64-atom cluster 4.28 -> 2.54 ms, 24 molecules 23.4 ->
// 11.9 ms, 304-atom slab 64.2 -> 32.8 ms; density of the cluster 0.67 -> 0.45 ms.
template <int MODE, int KS>  // MODE 0: density, 1: adjoint; KS: G' blocks per stage
__global__ void __launch_bounds__(kThreads, 1)
    k_split_rowdot(DevGrid G, const RdItem* __restrict__ items, int n_items, const double* __restrict__ scratch,
                   const int* __restrict__ rowexp, const unsigned char* __restrict__ gsl, unsigned present,
                   int weighted, double* __restrict__ out, double* __restrict__ part, unsigned* status) {
  using L = Layout<KS>;
  constexpr int kStages = L::kStages;
  extern __shared__ __align__(1024) unsigned char smem[];
  double* sY = reinterpret_cast<double*>(smem + L::kSmemY);  // [column half][point]
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kSmemBar);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::kSmemBar + L::kNumBars * 8);
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + L::kSmemBar + L::kNumBars * 8 + 4);

  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  const uint32_t smem0 = smem_u32(smem);
  if (smem0 & 127u) {  // operand tiles and bulk copies need aligned stages
    if (tid == 0) atomicOr(status, 2u);
    return;
  }
  const uint32_t bar0 = smem_u32(bars);
  auto slotfull_bar = [&](int k) { return bar0 + 8u * k; };
  auto slotempty_bar = [&](int k) { return bar0 + 8u * (kSlots + k); };
  auto gfull_bar = [&](int set, int k) { return bar0 + 8u * (2 * kSlots + set * kStages + k); };
  auto gempty_bar = [&](int set, int k) { return bar0 + 8u * (2 * kSlots + (2 + set) * kStages + k); };
  auto accfull_bar = [&](int k) { return bar0 + 8u * (2 * kSlots + 4 * kStages + k); };
  auto accempty_bar = [&](int k) { return bar0 + 8u * (2 * kSlots + 4 * kStages + 2 + k); };
  auto drain_bar = [&](int k) { return bar0 + 8u * (2 * kSlots + 4 * kStages + 4 + k); };

  if (tid == 0) {
    for (int k = 0; k < kSlots; ++k) {
      mbar_init(slotfull_bar(k), kSlicers);
      mbar_init(slotempty_bar(k), 2);  // both MMA warps
    }
    for (int k = 0; k < 2 * kStages; ++k) {
      mbar_init(gfull_bar(0, k), 1);
      mbar_init(gempty_bar(0, k), 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(accfull_bar(k), 1);
      mbar_init(accempty_bar(k), kEpiThreads);
      mbar_init(drain_bar(k), 1);
    }
    *s_abort = 0;
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = uniform(*tmem_slot);

  if (warp < kSlicers / 32) {
    // ---------------------------------------------------------- slicers
    const int r = warp * 32 + lane;  // point row
    const uint32_t dst0 = smem0 + (r >> 3) * kSBO + (r & 7) * 16;
    EntryWalk<MODE> W(items, n_items, present);
    float2 x[kKc];
    float mag = 0.f;
    bool live = false;
    int left = 0;  // functions from the chunk's first on
    int item = -1;
    float mq[MODE == 0 ? 1 : 4];  // rounding constants of the walk's current item per quantity
    // raw values of the walk's entry (zeros past the batch's functions and points)
    auto load = [&]() {
      const Item& I = W.I;
      const int p = I.pt * kPts + r;
      live = p < I.np;
      if (item != W.n) {
        item = W.n;
        int4 e = make_int4(-30000, -30000, -30000, -30000);
        if (live) e = *reinterpret_cast<const int4*>(rowexp + 4 * (I.bp0 + p));
        mq[0] = magic0(e.x - kFine);
        if constexpr (MODE == 1) {
          mq[1] = magic0(e.y - kFine);
          mq[2] = magic0(e.z - kFine);
          mq[3] = magic0(e.w - kFine);
        }
      }
      const int q = W.S.q, f0 = (W.S.c0 + W.e) * kKc;
      mag = mq[0];
      if constexpr (MODE == 1) mag = q == 0 ? mag : q == 1 ? mq[1] : q == 2 ? mq[2] : mq[3];
      // no load is conditional: functions past the batch's read the last one and
      // are cleared below, points past n_p the row's end (their rows are dropped)
      const float2* src = reinterpret_cast<const float2*>(scratch) + I.scr + q * I.plane + min(p, I.ldp - 1);
      left = I.nb - f0;
#pragma unroll
      for (int k = 0; k < kKc; ++k) x[k] = ldg_stream(src + static_cast<int64_t>(min(f0 + k, I.nb - 1)) * I.ldp);
    };
    int slot = 0, ph = 1;
    bool more = W.next();
    if (more) load();
    while (more) {
      if (!mbar_wait_warp(slotempty_bar(slot), ph, s_abort, status, G.wait_ns)) break;
      const uint32_t dst = dst0 + slot * kSlot;
      const bool store = __any_sync(0xffffffffu, live);  // a warp with no point leaves its rows as they are
      const float m = mag;
      if (left < kKc) {
#pragma unroll
        for (int k = 0; k < kKc; ++k)
          if (k >= left) x[k] = make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {  // functions 8h .. 8h + 7: one 16-byte row piece per digit
        uint32_t w[kSlices][4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          float2 d[kSlices];
          slice6x2(pk2(x[8 * h + 2 * u].x, x[8 * h + 2 * u + 1].x), pk2(x[8 * h + 2 * u].y, x[8 * h + 2 * u + 1].y),
                   m, d);
#pragma unroll
          for (int t = 0; t < kSlices; ++t) w[t][u] = bf16x2_exact(d[t]);
        }
        if (store) {
#pragma unroll
          for (int t = 0; t < kSlices; ++t)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + t * kDigA + h * kLBO), "r"(w[t][0]),
                         "r"(w[t][1]), "r"(w[t][2]), "r"(w[t][3])
                         : "memory");
        }
      }
      fence_async_smem();
      mbar_arrive(slotfull_bar(slot));
      if (++slot == kSlots) {
        slot = 0;
        ph ^= 1;
      }
      // the next entry's loads fly while its slot is awaited
      more = W.next();
      if (more) load();
    }
  } else if (warp >= kProdWarp) {
    // ---------------------------------------------------------- G' stream
    // A block takes its thread a few hundred clocks of barrier round trips, so
    // each ring has a producer of its own.
    const int set = warp - kProdWarp;
    int st = 0, ph = 1, k = 0, filled = 0;  // ring position and parity, groups, stages filled
    bool ok = true;
    GroupWalk<MODE> W(present);
    const uint32_t ring = smem0 + L::kSmemRing + set * kStages * L::kStage;
    for (int n = blockIdx.x; n < n_items && ok; n += gridDim.x) {
      W.open(items + n);
      // the next item's rows of F and R, fetched into L2 while this one runs:
      // its first readers would each wait for DRAM (only where all CTAs'
      // next items fit there beside the current ones)
      if (n + gridDim.x < n_items) {
        const Item N = item_of<MODE>(items + n + gridDim.x, present);
        const int rows = (MODE == 0 ? 1 : 4) * N.nb;
        if (N.nb <= 128) {
          const int p0 = N.pt * kPts;
          const uint32_t bytes = (min(kPts, N.ldp - p0) * 8);  // ldp is a multiple of 8: 64-byte pieces
          const float2* src = reinterpret_cast<const float2*>(scratch) + N.scr + p0;
          for (int f = 32 * set + lane; f < rows; f += 64)
            prefetch_l2(src + static_cast<int64_t>(f) * N.ldp, bytes);
        }
      }
      if (lane == 0) {
        const unsigned char* gb = gsl + W.I.gsl;
        for (; ok && W.next(); ++k) {
          if ((k & 1) != set) continue;
          const uint32_t blk = kSlices * kRowBytes * jt_width(W.I.nb, W.jt);
          const unsigned char* src = gb + (static_cast<int64_t>(W.m) * W.I.n_jt + W.jt) * W.I.n_ic * kBlockB +
                                     static_cast<int64_t>(W.S.c0) * blk;
          for (int c = 0; c < W.n; c += KS) {
            if (!mbar_wait_abort(gempty_bar(set, st), ph, s_abort, status, G.wait_ns)) {
              ok = false;
              break;
            }
            const uint32_t bytes = min(KS, W.n - c) * blk;
            arrive_expect_tx(gfull_bar(set, st), bytes);
            bulk_copy(ring + st * L::kStage, src, bytes, gfull_bar(set, st));
            src += bytes;
            ++filled;
            if (++st == kStages) {
              st = 0;
              ph ^= 1;
            }
          }
        }
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
    }
    // no copy outlives the CTA: the last kStages issued ones have landed
    if (lane == 0)
      for (int h = max(0, filled - kStages); h < filled; ++h)
        (void)mbar_wait(gfull_bar(set, h % kStages), (h / kStages) & 1, status);
    __syncwarp();
  } else if (warp == kMmaWarp || warp == kMmaWarp + 1) {
    // ---------------------------------------------------------- MMA issue
    // The whole warp walks and waits; one lane issues.  Operands of
    // tcgen05.mma are uniform registers: from values the compiler knows to be
    // the same in every lane an instruction issues in a few clocks, from a
    // single-lane loop each took about 200.  The tensor unit queues only a few
    // instructions, so what a warp does between its steps leaves it idle: two
    // warps issue, each the groups of one accumulator set, and one's
    // bookkeeping runs under the other's products.
    //
    // A wait by parity is only sound for a warp that has seen the barrier's
    // previous phase: each set has a ring of G' blocks of its own, and each
    // warp waits for every entry in order, also for those whose groups it
    // leaves to the other, before it gives the slot back.
    const int set = uniform(warp - kMmaWarp);
    int st = 0, ph = 0, k = 0, known = 0;  // ring position and parity, groups, entries seen in place
    bool ok = true;
    GroupWalk<MODE> W(present);
    const uint64_t descA = make_desc(smem0, kSBO);
    const uint64_t descB = make_desc(smem0 + L::kSmemRing + set * kStages * L::kStage, kSBO);
    const uint32_t t0 = uniform(tmem + set * kSetCols);
    auto see = [&](int e) {  // every entry up to e is in place
      for (; known <= e; ++known)
        if (!mbar_wait_warp(slotfull_bar(known % kSlots), (known / kSlots) & 1, s_abort, status, G.wait_ns))
          return false;
      return true;
    };
    for (int n = blockIdx.x; n < n_items && ok; n += gridDim.x) {
      W.open(items + n);
      for (; ok && W.next(); ++k) {
        if ((k & 1) != set) {  // the other warp's group
          if (W.last) {  // this warp is through with the segment's slots
            ok = see(W.ent + W.S.n - 1);
            if (ok && elect_one())
              for (int e = W.ent; e < W.ent + W.S.n; ++e) mma_commit(slotempty_bar(e % kSlots));
          }
          continue;
        }
        if (!mbar_wait_warp(accempty_bar(set), ((k >> 1) & 1) ^ 1, s_abort, status, G.wait_ns)) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (!see(W.ent + W.n - 1)) {  // every entry the group reads
          ok = false;
          break;
        }
        tc_fence_after();
        const int w = uniform(jt_width(W.I.nb, W.jt));
        for (int c = 0; c < W.n; c += KS) {
          if (!mbar_wait_warp(gfull_bar(set, st), ph, s_abort, status, G.wait_ns)) {
            ok = false;
            break;
          }
          tc_fence_after();
#pragma unroll
          for (int h = 0; h < KS; ++h) {
            if (c + h >= W.n) break;
            const int slot = uniform((W.ent + c + h) % kSlots);
            const uint64_t a = descA + static_cast<uint32_t>(slot * (kSlot >> 4));
            const uint64_t bd = descB + static_cast<uint32_t>((st * L::kStage + h * kSlices * kRowBytes * w) >> 4);
            if (elect_one()) {
              mma_row_levels(t0, a, bd, w, c + h == 0);
              if (W.last) mma_commit(slotempty_bar(slot));
            }
          }
          if (elect_one()) mma_commit(gempty_bar(set, st));
          if (++st == kStages) {
            st = 0;
            ph ^= 1;
          }
        }
        if (!ok) break;
        if (elect_one()) mma_commit(accfull_bar(set));
      }
    }
    // every MMA issued by this warp has completed before tensor memory is freed
    if (elect_one()) {
      mma_commit(drain_bar(set));
      (void)mbar_wait(drain_bar(set), 0, status);
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------- epilogue
    // Thread = one point; column group eg takes half of the group's columns
    const int eg = (warp - kEpiWarp0) >> 2;
    const int quarter = warp & 3;  // TMEM lanes 32 quarter .. +31
    const int r = quarter * 32 + lane;
    const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
    int k = 0;
    bool ok = true;
    GroupWalk<MODE> W(present);
    for (int n = blockIdx.x; n < n_items; n += gridDim.x) {
      W.open(items + n);
      const Item& I = W.I;
      const float2* base = reinterpret_cast<const float2*>(scratch) + I.scr;
      const int p = I.pt * kPts + r;
      const bool live = p < I.np;
      const bool busy = I.pt * kPts + quarter * 32 < I.np;  // some point of this warp exists
      df y = {0.f, 0.f};  // running sum over the item's groups
      // R of this thread's point and its 16 columns (8 in a 16-wide tile) of the
      // walk's group.  Columns past the batch's functions read the last one (their
      // U is zero), points past n_p the row's end (their result is dropped): no
      // load is conditional, so that all are in flight at once.
      const float2* mine = base + min(p, I.ldp - 1);
      auto load_R = [&](float2* R) {
        const int w = jt_width(I.nb, W.jt), j0 = W.jt * kTileJ + eg * (w >> 1);
        const float2* plane = mine + W.qr * I.plane;
#pragma unroll
        for (int i = 0; i < 8; ++i) R[i] = ldg_stream(plane + static_cast<int64_t>(min(j0 + i, I.nb - 1)) * I.ldp);
        if (w > 16) {
#pragma unroll
          for (int i = 8; i < 16; ++i) R[i] = ldg_stream(plane + static_cast<int64_t>(min(j0 + i, I.nb - 1)) * I.ldp);
        }
      };
      // values load one group ahead, across the item's groups
      float2 Rc[16], Rn[16];
      bool have = W.next();
      if (have && busy) load_R(Rc);
      while (have) {
        const int set = k & 1, w = jt_width(I.nb, W.jt);
        have = W.next();
        if (have && busy) load_R(Rn);
        ok = mbar_wait_warp(accfull_bar(set), (k >> 1) & 1, s_abort, status, G.wait_ns);
        if (!ok) break;
        tc_fence_after();
        // this group's sum yh + yl, even and odd columns apart (packed
        // instructions: the issue slots are shared with the slicers): per column
        // u = two-sums of the exact levels 0-2, the rounded levels and the errors
        // as its low part; the product with R = (rh, rl) keeps its FMA error
        // term unnormalised, and the sum adds each product by a two-sum whose
        // error joins yl
        float2 yh = {0.f, 0.f}, yl = {0.f, 0.f};
        if (busy) {
          const uint32_t t = tmem + lane_base + set * kSetCols + eg * (w >> 1);
#pragma unroll
          for (int c = 0; c < 16; c += 8) {
            if (c && w <= 16) break;
            float v[6][8];
            tmem_ld8x6(t + c, w, v);
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
              float2 s, es, u, eu, a, ea;
              two_sum2(pk2(v[0][i], v[0][i + 1]), pk2(v[1][i], v[1][i + 1]), s, es);
              two_sum2(s, pk2(v[2][i], v[2][i + 1]), u, eu);
              const float2 ul = add2(add2(es, eu), add2(pk2(v[3][i], v[3][i + 1]),
                                                        add2(pk2(v[4][i], v[4][i + 1]), pk2(v[5][i], v[5][i + 1]))));
              const float2 rh = pk2(Rc[c + i].x, Rc[c + i + 1].x), rl = pk2(Rc[c + i].y, Rc[c + i + 1].y);
              const float2 ph = mul2(rh, u);
              float2 pl = fma2(rh, u, pk2(-ph.x, -ph.y));
              pl = fma2(rh, ul, pl);
              pl = fma2(rl, u, pl);
              two_sum2(yh, ph, a, ea);
              yh = a;
              yl = add2(yl, add2(ea, pl));
            }
          }
        }
        tc_fence_before();
        mbar_arrive(accempty_bar(set));
        ++k;
        y = df_add(y, df_add(df{yh.x, yl.x}, df{yh.y, yl.y}));
#pragma unroll
        for (int i = 0; i < 16; ++i) Rc[i] = Rn[i];
      }
      // the two column halves of each point (a warp that gave up ends them all)
      sY[eg * kPts + r] = static_cast<double>(y.hi) + static_cast<double>(y.lo);
      if (bar_red_or(2, kEpiThreads, !ok)) break;
      if (eg == 0 && live) {
        const double val = sY[r] + sY[kPts + r];
        const int64_t gp = I.bp0 + p;
        if (I.part < 0)
          out[gp] = weighted ? G.w[gp] * val : val;
        else
          part[I.part * kPts + r] = val;  // a share of the batch's j-tiles: k_rowdot_sum adds them up
      }
      bar_sync(2, kEpiThreads);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

// The points of tiles whose j-tiles were shared out: their shares' sums added in
// order (one CTA per tile; 8 bytes a share and point, 20 MB for the 304-atom slab).
__global__ void __launch_bounds__(kPts) k_rowdot_sum(const RdSum* __restrict__ sums, const double* __restrict__ part,
                                                   const double* __restrict__ w, int weighted,
                                                   double* __restrict__ out) {
  const RdSum s = sums[blockIdx.x];
  const int r = threadIdx.x;
  if (r >= s.n) return;
  const double* x = part + static_cast<int64_t>(s.slot0) * kPts + r;
  double y = x[0];
  for (int k = 1; k < s.shares; ++k) y += x[k * kPts];
  out[s.pt0 + r] = weighted ? w[s.pt0 + r] * y : y;
}

// the prepared matrices of one call: FP32-pair copies in slots [slot, slot + 5)
// of the grid's buffer and their column bounds per block; slot 0 for the density,
// 5 for the adjoint.  Returns the mask of present matrices.
q4c_status prepare(const q4c_grid* g, const double* const mats[5], int slot, unsigned* present, cudaStream_t s) {
  int dev = 0, n_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  *present = 0;
  if (g->nnz == 0) return Q4C_OK;
  Mats M;
  for (int m = 0; m < 5; ++m) {
    M.m[m] = mats[m];
    if (mats[m]) *present |= 1u << m;
  }
  const size_t smem = sizeof(unsigned) * 5 * *std::max_element(g->tables->nfn.begin(), g->tables->nfn.end());
  if (smem > 12 * 1024)
    Q4C_CUDA(cudaFuncSetAttribute(k_prepare_blocks, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
  KernelScope ks("split_gslice", s);
  const unsigned nblk = static_cast<unsigned>(std::min<int64_t>(g->n_blocks, 64 * n_sm));
  k_prepare_blocks<<<nblk, 128, smem, s>>>(g->tables->view(), g->view(), M, g->n_blocks, g->d_blk_row, g->d_blk_col,
                                           g->d_blk_off, g->d_blk_T, g->d_cm_off, g->d_gdf + slot * g->nnz, g->nnz,
                                           g->d_cm + slot * g->cm_total, g->cm_total);
  Q4C_CUDA(cudaGetLastError());
  return Q4C_OK;
}

// G' digit blocks of one wave [b0, b1); the wave's offset tables must be in place
template <int MODE>
q4c_status gslice_wave(const q4c_grid* g, int wv, int slot, unsigned present, cudaStream_t s) {
  const int64_t b0 = g->wave_b0[wv], b1 = g->wave_b0[wv + 1];
  if (b1 <= b0 || present == 0) return Q4C_OK;
  // two j-tiles a CTA: the batches of a wave differ widely in n_b
  const unsigned y = static_cast<unsigned>(std::max(1, (g->max_nb + 2 * kTileJ - 1) / (2 * kTileJ)));
  KernelScope ks("split_gslice", s);
  k_gslice<MODE == 0 ? 1 : 5><<<dim3(static_cast<unsigned>(b1 - b0), y), 256, 0, s>>>(
      g->view(), b0, g->d_gdf + slot * g->nnz, g->nnz, present, g->d_cm + slot * g->cm_total, g->cm_total,
      g->d_pair_blk, g->d_cm_off, g->d_gsl_off, reinterpret_cast<uint32_t*>(g->d_gsl));
  Q4C_CUDA(cudaGetLastError());
  return Q4C_OK;
}

// the row-dot kernel of one wave (its G' blocks in place)
template <int MODE, int KS>
q4c_status rowdot_kernel(const q4c_grid* g, int wv, unsigned present, bool weighted, double* out, cudaStream_t s,
                         const char* name) {
  int dev = 0, n_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  Q4C_CUDA(cudaFuncSetAttribute(k_split_rowdot<MODE, KS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                Layout<KS>::kSmemTotal));
  const int64_t i0 = g->rd_w0[wv], i1 = g->rd_w0[wv + 1];
  const int n_items = static_cast<int>(i1 - i0);
  if (n_items == 0) return Q4C_OK;
  const int grid = std::min(n_items, n_sm);
  {
    KernelScope ks(name, s);
    k_split_rowdot<MODE, KS><<<grid, kThreads, Layout<KS>::kSmemTotal, s>>>(
        g->view(), g->d_rd_items + i0, n_items, g->d_scratch, g->d_rowexp,
        reinterpret_cast<const unsigned char*>(g->d_gsl), present, weighted ? 1 : 0, out, g->d_rd_part, g->d_status);
  }
  Q4C_CUDA(cudaGetLastError());
  const int64_t s0 = g->rd_s0[wv], s1 = g->rd_s0[wv + 1];
  if (s1 > s0) {
    KernelScope ks("split_rowdot_sum", s);
    k_rowdot_sum<<<static_cast<unsigned>(s1 - s0), kPts, 0, s>>>(g->d_rd_sums + s0, g->d_rd_part, g->d_w,
                                                                 weighted ? 1 : 0, out);
    Q4C_CUDA(cudaGetLastError());
  }
  return Q4C_OK;
}

template <int MODE>
q4c_status kernel_ks(const q4c_grid* g, int wv, unsigned present, bool weighted, double* out, cudaStream_t s, int ks,
                     const char* name) {
  if (ks == 2) return rowdot_kernel<MODE, 2>(g, wv, present, weighted, out, s, name);
  return rowdot_kernel<MODE, 1>(g, wv, present, weighted, out, s, name);
}

template <int MODE>
q4c_status wave(const q4c_grid* g, int wv, int slot, unsigned present, bool weighted, double* out, cudaStream_t s) {
  if (g->wave_b0[wv + 1] <= g->wave_b0[wv]) return Q4C_OK;
  if (q4c_status st = gslice_wave<MODE>(g, wv, slot, present, s)) return st;
  return kernel_ks<MODE>(g, wv, present, weighted, out, s, g->rd_ks, MODE == 0 ? "split_density" : "split_backward");
}

template <int MODE>
q4c_status run(const q4c_tables* t, const q4c_grid* g, const double* const mats[5], double* out, cudaStream_t s,
               bool weighted) {
  if (g->max_nb > kMaxNb) {
    set_error("the split density/adjoint need at most 4096 active functions per batch");
    return Q4C_EUNSUPPORTED;
  }
  unsigned present = 0;
  if (q4c_status st = prepare(g, mats, 0, &present, s)) return st;
  const int n_waves = static_cast<int>(g->wave_b0.size()) - 1;
  for (int wv = 0; wv < n_waves; ++wv) {
    const int64_t b0 = g->wave_b0[wv], b1 = g->wave_b0[wv + 1];
    if (b1 <= b0) continue;
    if (q4c_status st = launch_fill_idx(t, g, b0, b1, s)) return st;
    if (q4c_status st = launch_basis_df(t, g, b0, b1, nullptr, nullptr, g->d_rowexp, MODE == 0 ? 1 : 4, s)) return st;
    if (q4c_status st = wave<MODE>(g, wv, 0, present, weighted, out, s)) return st;
  }
  return Q4C_OK;
}

}  // namespace rowdot

q4c_status rowdot_prepare(const q4c_grid* g, const double* const mats[5], int slot, unsigned* present,
                          cudaStream_t s) {
  return rowdot::prepare(g, mats, slot, present, s);
}

q4c_status rowdot_wave(const q4c_grid* g, int wv, int mode, int slot, unsigned present, bool weighted, double* out,
                       cudaStream_t s) {
  return mode == 0 ? rowdot::wave<0>(g, wv, slot, present, weighted, out, s)
                   : rowdot::wave<1>(g, wv, slot, present, weighted, out, s);
}

// the tuner's part for the row-dot kernel: the adjoint kernel of wave 0 with
// both stage shapes (G' from zero matrices, sliced once: the kernel's work
// does not depend on the values), one untimed launch each, then three rounds
// alternating the shapes, each launch between CUDA events; the faster shape
// is kept for the grid.  The wave's offset tables and basis tiles with
// per-point exponents must be in place.
q4c_status autotune_rowdot(q4c_grid* g, double* out, cudaStream_t s) {
  g->rd_tune_ms[0] = g->rd_tune_ms[1] = -1.0;
  if (g->wave_b0.size() < 2 || g->max_nb > rowdot::kMaxNb || g->nnz == 0) return Q4C_OK;
  if (g->wave_b0[1] <= g->wave_b0[0]) return Q4C_OK;
  Q4C_CUDA(cudaMemsetAsync(g->d_gdf + 5 * g->nnz, 0, sizeof(float2) * 5 * g->nnz, s));
  Q4C_CUDA(cudaMemsetAsync(g->d_cm + 5 * g->cm_total, 0, sizeof(float) * 5 * g->cm_total, s));
  if (q4c_status st = rowdot::gslice_wave<1>(g, 0, 5, 31u, s)) return st;
  cudaEvent_t ev[2][3][2] = {};
  q4c_status status = Q4C_OK;
  for (int k = 0; k < 2; ++k)
    for (int r = 0; r < 3; ++r)
      for (int e = 0; e < 2; ++e)
        if (cudaEventCreate(&ev[k][r][e]) != cudaSuccess) status = Q4C_ECUDA;
  for (int ks = 1; ks <= 2 && status == Q4C_OK; ++ks)
    status = rowdot::kernel_ks<1>(g, 0, 31u, true, out, s, ks, "split_tune");
  for (int r = 0; r < 3 && status == Q4C_OK; ++r)
    for (int ks = 1; ks <= 2 && status == Q4C_OK; ++ks) {
      cudaEventRecord(ev[ks - 1][r][0], s);
      status = rowdot::kernel_ks<1>(g, 0, 31u, true, out, s, ks, "split_tune");
      cudaEventRecord(ev[ks - 1][r][1], s);
    }
  if (status == Q4C_OK && cudaStreamSynchronize(s) != cudaSuccess) status = Q4C_ECUDA;
  for (int k = 0; k < 2 && status == Q4C_OK; ++k) {
    double sum = 0.0;
    for (int r = 0; r < 3; ++r) {
      float ms = 0.f;
      if (cudaEventElapsedTime(&ms, ev[k][r][0], ev[k][r][1]) != cudaSuccess) status = Q4C_ECUDA;
      sum += ms;
    }
    g->rd_tune_ms[k] = sum / 3.0;
  }
  if (status == Q4C_OK) g->rd_ks = g->rd_tune_ms[1] < g->rd_tune_ms[0] ? 2 : 1;
  else set_error("q4c_autotune: timing of the density/adjoint kernel failed");
  for (int k = 0; k < 2; ++k)
    for (int r = 0; r < 3; ++r)
      for (int e = 0; e < 2; ++e)
        if (ev[k][r][e]) cudaEventDestroy(ev[k][r][e]);
  return status;
}

q4c_status density_split(const q4c_tables* t, const q4c_grid* g, const double* P, double* n, cudaStream_t s) {
  const double* mats[5] = {P, nullptr, nullptr, nullptr, nullptr};
  return rowdot::run<0>(t, g, mats, n, s, false);
}

q4c_status backward_split(const q4c_tables* t, const q4c_grid* g, const q4c_matrices* Gm, double* dLdv,
                          cudaStream_t s, bool weighted) {
  const double* mats[5] = {Gm->V, Gm->W0, Gm->SOx, Gm->SOy, Gm->SOz};
  // with every slot NULL the gradient is zero
  if (!Gm->V && !Gm->W0 && !Gm->SOx && !Gm->SOy && !Gm->SOz) {
    Q4C_CUDA(cudaMemsetAsync(dLdv, 0, sizeof(double) * g->n_pts, s));
    return Q4C_OK;
  }
  return rowdot::run<1>(t, g, mats, dLdv, s, weighted);
}

}  // namespace q4c
