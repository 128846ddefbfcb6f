// Plain FP64 path: basis tiles per batch, batch products on the FP64 ALUs,
// FP64 atomic scatter into the block pattern, mirror, spinor assembly,
// density (Eqs. 39-40) and the adjoint.  This is the reference-precision GPU
// path the split-precision tensor-core path is measured against.
#include "basis.cuh"
#include "internal.h"

namespace q4c {

// ------------------------------------------------------------------ basis
// Tiles of batch b in the scratch wave: Phi, X, Y, Z each [n_b][ldp],
// ldp = n_p rounded up to 8; one thread per (point, active atom).
// With colexp != NULL (split path) it also records, per batch and local
// function, binary exponents e with |value| < 2^e for the unscaled sets
// (Phi, X, Y, Z: slots 4..7) and upper bounds for the D-scaled sets
// (D = w v; slots 0..3, from e(D_p) + e(value)), colexp[8 n_b] per batch.
__device__ __forceinline__ int binexp(double x) {  // |x| < 2^binexp(x), x != 0
  const int E = static_cast<int>((__double_as_longlong(x) >> 52) & 0x7FF);
  return E - 1022;
}
constexpr int kNoExp = -30000;
// scr_base: subtracted from the batch offsets (the first offset of a sub-wave
// whose tiles start at `scratch`; 0 for the grid's own workspace)
__global__ void k_basis_tiles(DevBasis B, DevGrid G, int64_t b0, const int64_t* __restrict__ scr_off,
                              int64_t scr_base, double* __restrict__ scratch, const double* __restrict__ v,
                              int* __restrict__ colexp) {
  extern __shared__ int s_exp[];  // [8][nb] when colexp != NULL
  const int64_t b = b0 + blockIdx.x;
  const int64_t p0 = G.pt_ptr[b];
  const int np = static_cast<int>(G.pt_ptr[b + 1] - p0);
  const int ldp = (np + 7) & ~7;
  const int a0 = G.bat_atom_ptr[b], na = G.bat_atom_ptr[b + 1] - a0;
  const int nb = static_cast<int>(G.bat_fn_ptr[b + 1] - G.bat_fn_ptr[b]);
  double* base = scratch + (scr_off[b] - scr_base);
  const int64_t plane = static_cast<int64_t>(nb) * ldp;
  if (colexp) {
    for (int i = threadIdx.x; i < 8 * nb; i += blockDim.x) s_exp[i] = kNoExp;
    __syncthreads();
  }
  for (int item = threadIdx.x; item < np * na; item += blockDim.x) {
    const int a = item / np, p = item - a * np;
    const int A = G.bat_atoms[a0 + a];
    const int f0 = G.bat_atom_fn0[a0 + a];
    const double dx = G.x[p0 + p] - G.c_xyz[3 * A], dy = G.y[p0 + p] - G.c_xyz[3 * A + 1],
                 dz = G.z[p0 + p] - G.c_xyz[3 * A + 2];
    int eD = kNoExp;
    if (colexp) {
      const double D = G.w[p0 + p] * v[p0 + p];
      if (D != 0.0) eD = binexp(D);
    }
    atom_functions(B, G.c_sp[A], dx, dy, dz, [&](int k, double phi, double gx, double gy, double gz) {
      double* q = base + static_cast<int64_t>(f0 + k) * ldp + p;
      q[0] = phi;
      q[plane] = gx;
      q[2 * plane] = gy;
      q[3 * plane] = gz;
      if (colexp) {
        const double vals[4] = {phi, gx, gy, gz};
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          if (vals[s] == 0.0) continue;
          const int e = binexp(vals[s]);
          atomicMax(&s_exp[(4 + s) * nb + f0 + k], e);
          if (eD != kNoExp) atomicMax(&s_exp[s * nb + f0 + k], e + eD);
        }
      }
    });
  }
  if (colexp) {
    __syncthreads();
    int* out = colexp + 8 * G.bat_fn_ptr[b];
    for (int i = threadIdx.x; i < 8 * nb; i += blockDim.x) out[i] = s_exp[i];
  }
}

q4c_status launch_basis_tiles(const q4c_tables* t, const q4c_grid* g, int64_t b0, int64_t b1, const double* v,
                              int* colexp, cudaStream_t s) {
  const size_t smem = colexp ? sizeof(int) * 8 * std::max(g->max_nb, 1) : 0;
  if (smem > 48 * 1024)
    Q4C_CUDA(cudaFuncSetAttribute(k_basis_tiles, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
  KernelScope ks("basis", s);
  k_basis_tiles<<<static_cast<unsigned>(b1 - b0), 256, smem, s>>>(t->view(), g->view(), b0, g->d_scr_off, 0,
                                                                   g->d_scratch, v, colexp);
  Q4C_CUDA(cudaGetLastError());
  return Q4C_OK;
}

// nf of the atom behind local atom a of a batch
__device__ __forceinline__ int local_nf(const DevBasis& B, const DevGrid& G, int a0, int a) {
  return __ldg(B.sp_nfn + G.c_sp[G.bat_atoms[a0 + a]]);
}

// ------------------------------------------------------------ products
// One CTA per 32x32 tile (ti <= tj) of one batch: V, W0 and SO of its pairs
// i <= j, scattered with FP64 atomics into the upper blocks.
// The FP64 units (2 multiply-adds a clock and SM) bound it: 10 multiply-adds
// per pair and point.  So only pairs that count are formed, in blocks of 4 x 4
// (eight lanes each, two pairs a lane; a warp takes four blocks of the tile's
// list): blocks wholly below the diagonal or past the batch's functions are left
// out, and the points run to n_p, not to a multiple of the staged 16.  The
// groups of four blocks are dealt to the warps starting at a warp that rotates
// with the CTA, so that the four schedulers' FP64 units get equal shares over
// the CTAs of an SM.  gridDim.y splits a batch's points where a wave has too
// few tiles to fill the GPU (the partial sums meet in the scatter's atomics).
// 64-atom cluster (5.5e9 n_p n_b^2): 91.6 ms with whole 32x32 tiles, 56.2 with
// blocks of 8 x 8 -> 51.9; water (24 functions): 223 us -> 81.
constexpr int kT = 32, kK = 16;
constexpr int kPitch = kK + 1;  // doubles per staged function: rows fall into distinct banks
constexpr int kSub = 4;         // side of a block of pairs
__global__ void __launch_bounds__(256, 3) k_products_fp64(DevBasis B, DevGrid G, const int4* __restrict__ tiles,
                                                       int64_t t0, const int64_t* __restrict__ scr_off,
                                                       int64_t scr_base, const double* __restrict__ scratch,
                                                       const double* __restrict__ v, double* V, double* W0,
                                                       double* SOx, double* SOy, double* SOz) {
  __shared__ double sa[4][kT][kPitch];  // D-scaled i side
  __shared__ double sb[4][kT][kPitch];  // j side
  const int4 tile = tiles[t0 + blockIdx.x];
  const int64_t b = tile.x;
  const int ti = tile.y, tj = tile.z;
  const int64_t p0 = G.pt_ptr[b];
  const int n_pt = static_cast<int>(G.pt_ptr[b + 1] - p0);
  const int ldp = (n_pt + 7) & ~7;
  const int share = ((n_pt + gridDim.y - 1) / gridDim.y + kK - 1) & ~(kK - 1);  // points of this CTA: [kb, np)
  const int kb = blockIdx.y * share, np = min(n_pt, kb + share);
  if (kb >= np) return;
  const int nb = static_cast<int>(G.bat_fn_ptr[b + 1] - G.bat_fn_ptr[b]);
  const int64_t plane = static_cast<int64_t>(nb) * ldp;
  const double* base = scratch + (scr_off[b] - scr_base);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // this warp's two groups of four blocks, one block for each eight lanes:
  // first row and column of the lane's block, -1 for none
  int ri[2], cj[2];
  bool any[2];
  {
    const int nr = (min(kT, nb - ti * kT) + kSub - 1) / kSub, nc = (min(kT, nb - tj * kT) + kSub - 1) / kSub;
    const int n_blk = ti == tj ? nr * (nr + 1) / 2 : nr * nc;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int first = 4 * (((warp + blockIdx.x) & 7) + 8 * u);
      int k = first + (lane >> 3);
      any[u] = first < n_blk;
      ri[u] = cj[u] = -1;
      if (k < n_blk) {
        int r = 0;
        if (ti == tj) {
          while (k >= nc - r) k -= nc - r++;
          k += r;
        } else {
          r = k / nc;
          k -= r * nc;
        }
        ri[u] = r * kSub + ((lane >> 1) & 3);
        cj[u] = k * kSub + 2 * (lane & 1);
      }
    }
  }
  double acc[2][2][5];
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int w = 0; w < 2; ++w)
#pragma unroll
      for (int q = 0; q < 5; ++q) acc[u][w][q] = 0.0;

  for (int k0 = kb; k0 < np; k0 += kK) {
    __syncthreads();
    {  // thread: point kk of the functions f, f + 16 of both sides
      const int kk = threadIdx.x & (kK - 1), p = k0 + kk;
      const double d = p < np ? G.w[p0 + p] * v[p0 + p] : 0.0;
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int f = (threadIdx.x >> 4) + 16 * h;
          const int fi = ti * kT + f, fj = tj * kT + f;
          const double bj = (p < np && fj < nb) ? base[q * plane + static_cast<int64_t>(fj) * ldp + p] : 0.0;
          double ai = bj;
          if (ti != tj) ai = (p < np && fi < nb) ? base[q * plane + static_cast<int64_t>(fi) * ldp + p] : 0.0;
          sa[q][f][kk] = ai * d;
          sb[q][f][kk] = bj;
        }
    }
    __syncthreads();
    const int n_kk = min(kK, np - k0);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (!any[u]) continue;
      const int i = max(ri[u], 0), j = max(cj[u], 0);
#pragma unroll 4
      for (int kk = 0; kk < n_kk; ++kk) {
        double a[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = sa[q][i][kk];
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          double c[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) c[q] = sb[q][j + w][kk];
          acc[u][w][0] = fma(a[0], c[0], acc[u][w][0]);
          acc[u][w][1] = fma(a[1], c[1], fma(a[2], c[2], fma(a[3], c[3], acc[u][w][1])));
          acc[u][w][2] = fma(a[2], c[3], fma(-a[3], c[2], acc[u][w][2]));
          acc[u][w][3] = fma(a[3], c[1], fma(-a[1], c[3], acc[u][w][3]));
          acc[u][w][4] = fma(a[1], c[2], fma(-a[2], c[1], acc[u][w][4]));
        }
      }
    }
  }
  // scatter the upper triangle
  const int64_t f0 = G.bat_fn_ptr[b];
  const int a0 = G.bat_atom_ptr[b], na = G.bat_atom_ptr[b + 1] - a0;
  const int64_t pp = G.bat_pair_ptr[b];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (ri[u] < 0) continue;
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int i = ti * kT + ri[u], j = tj * kT + cj[u] + w;
      if (i >= nb || j >= nb || i > j) continue;
      const int ii = G.fn_info[f0 + i], jj = G.fn_info[f0 + j];
      const int ai = ii >> 16, ki = ii & 0xffff, aj = jj >> 16, kj = jj & 0xffff;
      const int64_t off = G.pair_off[pp + static_cast<int64_t>(ai) * na + aj];
      if (off < 0) continue;
      const int64_t e = off + static_cast<int64_t>(ki) * local_nf(B, G, a0, aj) + kj;
      atomicAdd(V + e, acc[u][w][0]);
      atomicAdd(W0 + e, acc[u][w][1]);
      if (i != j) {
        atomicAdd(SOx + e, acc[u][w][2]);
        atomicAdd(SOy + e, acc[u][w][3]);
        atomicAdd(SOz + e, acc[u][w][4]);
      }
    }
  }
}

// ------------------------------------------------- mirror + spinor blocks
// One CTA per block.  The batch kernels accumulate only the canonical half
// of the pattern: local functions are ordered by centre (cell, atom) with the
// cells lexicographic in T, so a pair i <= j always lands in a block (A, B, T)
// with T > 0, or T = 0 and A <= B.  Canonical blocks (role 1) are copied
// transposed into their partner (B, A, -T) (negated for SO); a block that is
// its own partner (A = B, T = 0; role 2) fills i > j from (j, i); role 0
// blocks are the copy targets.
// SPINOR: also the spinor blocks of both (k_spinor), from the same read.
template <bool SPINOR>
__global__ void k_mirror(const int* __restrict__ blk_row, const int* __restrict__ blk_col,
                         const int* __restrict__ blk_T, const int* __restrict__ blk_role,
                         const int64_t* __restrict__ blk_off, const int* atom_sp, const int* sp_nfn, double* V,
                         double* W0, double* SOx, double* SOy, double* SOz, double2* __restrict__ SS) {
  const int q = blockIdx.x;
  const int role = blk_role[q], A = blk_row[q], Bc = blk_col[q];
  const int64_t o = blk_off[q], oT = role ? blk_off[blk_T[q]] : 0;
  if (role == 0) return;
  const int nfA = sp_nfn[atom_sp[A]], nfB = sp_nfn[atom_sp[Bc]];
  const bool self = role == 2;
  auto spinor = [&](int64_t off, int nf, int i, int j, double w, double x, double y, double z) {
    double2* r0 = SS + 4 * off + static_cast<int64_t>(2 * i) * (2 * nf) + 2 * j;
    double2* r1 = r0 + 2 * nf;
    r0[0] = make_double2(w, z);
    r0[1] = make_double2(y, x);
    r1[0] = make_double2(-y, x);
    r1[1] = make_double2(w, -z);
  };
  for (int e = threadIdx.x; e < nfA * nfB; e += blockDim.x) {
    const int i = e / nfB, j = e - i * nfB;
    if (self && i > j) continue;
    const double v = V[o + e], w = W0[o + e], x = SOx[o + e], y = SOy[o + e], z = SOz[o + e];
    if (SPINOR) spinor(o, nfB, i, j, w, x, y, z);
    if (self && i == j) continue;
    const int64_t dst = oT + static_cast<int64_t>(j) * nfA + i;  // oT = o where the block is its own partner
    V[dst] = v;
    W0[dst] = w;
    SOx[dst] = -x;
    SOy[dst] = -y;
    SOz[dst] = -z;
    if (SPINOR) spinor(oT, nfA, j, i, w, -x, -y, -z);
  }
}

// [[W0 + i SOz, SOy + i SOx], [-SOy + i SOx, W0 - i SOz]] per element
__global__ void k_spinor(const int* __restrict__ blk_row, const int* __restrict__ blk_col,
                         const int64_t* __restrict__ blk_off, const int* atom_sp, const int* sp_nfn,
                         const double* __restrict__ W0, const double* __restrict__ SOx,
                         const double* __restrict__ SOy, const double* __restrict__ SOz, double2* __restrict__ SS) {
  const int q = blockIdx.x;
  const int nfB = sp_nfn[atom_sp[blk_col[q]]];
  const int nfA = sp_nfn[atom_sp[blk_row[q]]];
  const int64_t o = blk_off[q];
  for (int e = threadIdx.x; e < nfA * nfB; e += blockDim.x) {
    const int i = e / nfB, j = e - i * nfB;
    const double w = W0[o + e], x = SOx[o + e], y = SOy[o + e], z = SOz[o + e];
    double2* r0 = SS + 4 * o + static_cast<int64_t>(2 * i) * (2 * nfB) + 2 * j;
    double2* r1 = r0 + 2 * nfB;
    r0[0] = make_double2(w, z);
    r0[1] = make_double2(y, x);
    r1[0] = make_double2(-y, x);
    r1[1] = make_double2(w, -z);
  }
}

q4c_status mirror_and_spinor(const q4c_grid* g, const q4c_matrices* out, cudaStream_t s) {
  const q4c_tables* t = g->tables;
  if (g->n_blocks == 0) return Q4C_OK;
  auto launch = [&](auto kern) {
    KernelScope ks("mirror", s);
    kern<<<static_cast<unsigned>(g->n_blocks), 128, 0, s>>>(
        g->d_blk_row, g->d_blk_col, g->d_blk_T, g->d_blk_role, g->d_blk_off, g->d_atom_sp, t->d_sp_nfn, out->V,
        out->W0, out->SOx, out->SOy, out->SOz, reinterpret_cast<double2*>(out->spinor_SS));
  };
  // The transposed block's spinors leave 32 bytes at a time: with everything in the
  // L2 cache that is cheaper than a second launch and read (one molecule of 3 atoms:
  // 8 us for 14; 64-atom cluster, 0.2M elements: 19 us for 29), with a pattern of 19M
  // elements it is not (304-atom slab: 1.12 ms for 0.85).
  if (out->spinor_SS && g->nnz <= 1 << 20) {
    launch(k_mirror<true>);
    Q4C_CUDA(cudaGetLastError());
    return Q4C_OK;
  }
  launch(k_mirror<false>);
  Q4C_CUDA(cudaGetLastError());
  if (out->spinor_SS) {
    KernelScope ks("spinor", s);
    k_spinor<<<static_cast<unsigned>(g->n_blocks), 128, 0, s>>>(
        g->d_blk_row, g->d_blk_col, g->d_blk_off, g->d_atom_sp, t->d_sp_nfn, out->W0, out->SOx, out->SOy,
        out->SOz, reinterpret_cast<double2*>(out->spinor_SS));
    Q4C_CUDA(cudaGetLastError());
  }
  return Q4C_OK;
}

// the products of one wave (its basis tiles in place)
q4c_status products_fp64_wave(const q4c_grid* g, int wv, const double* v, const q4c_matrices* out,
                              cudaStream_t s) {
  const int64_t t0 = g->wave_t0[wv], t1 = g->wave_t0[wv + 1];
  if (t1 <= t0) return Q4C_OK;
  // fewer than eight CTAs a SM: split each batch's points, into no less than
  // 32 (a CTA's scatter then still costs less than its sums)
  int dev = 0, n_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  const int64_t want = (8ll * n_sm + t1 - t0 - 1) / (t1 - t0);
  const unsigned split = static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>(want, g->max_np / 32)));
  KernelScope ks("products_fp64", s);
  k_products_fp64<<<dim3(static_cast<unsigned>(t1 - t0), split), 256, 0, s>>>(g->tables->view(), g->view(), g->d_tiles, t0,
                                                                   g->d_scr_off, 0, g->d_scratch, v, out->V,
                                                                   out->W0, out->SOx, out->SOy, out->SOz);
  Q4C_CUDA(cudaGetLastError());
  return Q4C_OK;
}

q4c_status integrate_fp64(const q4c_tables* t, const q4c_grid* g, const double* v, const q4c_matrices* out,
                          cudaStream_t s) {
  double* outs[5] = {out->V, out->W0, out->SOx, out->SOy, out->SOz};
  for (double* o : outs) Q4C_CUDA(cudaMemsetAsync(o, 0, sizeof(double) * g->nnz, s));
  for (size_t wv = 0; wv + 1 < g->wave_b0.size(); ++wv) {
    const int64_t b0 = g->wave_b0[wv], b1 = g->wave_b0[wv + 1];
    if (b1 > b0) {
      if (q4c_status st = launch_basis_tiles(t, g, b0, b1, nullptr, nullptr, s)) return st;
    }
    if (q4c_status st = products_fp64_wave(g, static_cast<int>(wv), v, out, s)) return st;
  }
  return mirror_and_spinor(g, out, s);
}

// ------------------------------------------------------ per-column operator
// Eq. 19 in the scalar form of the large component: every element carries
// the eigenvalue and defining potential of its COLUMN's radial function,
//   F_ij = sum_p phi_i(p) theta_pj,  theta_pj = w_p (v_p + eps_j - V_j(|p - R_j|)) phi_j(p),
// so F is not symmetric: one CTA per 32x32 tile over all tile pairs of a
// batch, the column factors built while loading the j side, every element
// scattered (no mirror).  V_j: cubic in the knot index on each interval,
// the first knot's value below r_min and the last one's from r_c on.
__device__ __forceinline__ double column_potential(const DevBasis& B, const double* __restrict__ vcoef, int rad,
                                                   double r) {
  const double* c = vcoef + static_cast<int64_t>(rad) * (B.n_log - 1) * 4;
  if (r < B.r_min) return c[0];
  if (r >= B.r_c) {
    const double* e = c + (B.n_log - 2) * 4;
    return e[0] + e[1] + e[2] + e[3];
  }
  const double t = log(r * B.inv_rmin) * B.inv_h;
  const int k = min(max(static_cast<int>(t), 0), B.n_log - 2);
  const double s = t - k;
  const double* e = c + k * 4;
  return e[0] + s * (e[1] + s * (e[2] + s * e[3]));
}

__global__ void __launch_bounds__(256) k_columns_fp64(DevBasis B, DevGrid G, const int4* __restrict__ tiles,
                                                      const int64_t* __restrict__ scr_off,
                                                      const double* __restrict__ scratch,
                                                      const double* __restrict__ v, const double* __restrict__ eps,
                                                      const double* __restrict__ vcoef, double* F) {
  __shared__ double sa[kK][kT], sb[kK][kT];
  __shared__ double s_c[3][kT], s_eps[kT];
  __shared__ int s_rad[kT];
  const int4 tile = tiles[blockIdx.x];
  const int64_t b = tile.x;
  const int ti = tile.y, tj = tile.z;
  const int64_t p0 = G.pt_ptr[b];
  const int np = static_cast<int>(G.pt_ptr[b + 1] - p0);
  const int ldp = (np + 7) & ~7;
  const int64_t f0 = G.bat_fn_ptr[b];
  const int nb = static_cast<int>(G.bat_fn_ptr[b + 1] - f0);
  const int a0 = G.bat_atom_ptr[b], na = G.bat_atom_ptr[b + 1] - a0;
  const double* base = scratch + scr_off[b];
  if (threadIdx.x < kT) {  // centre, radial and eigenvalue of each column function of the tile
    const int fj = tj * kT + threadIdx.x;
    int rad = -1;
    if (fj < nb) {
      const int info = G.fn_info[f0 + fj];
      const int c = G.bat_atoms[a0 + (info >> 16)], k = info & 0xffff;
      const int sp = G.c_sp[c], r0 = __ldg(B.sp_rad0 + sp), nr = __ldg(B.sp_nrad + sp);
      for (int q = 0, first = 0; q < nr; ++q) {
        const int n = 2 * __ldg(B.rad_l + r0 + q) + 1;
        if (k < first + n) {
          rad = r0 + q;
          break;
        }
        first += n;
      }
      s_c[0][threadIdx.x] = G.c_xyz[3 * c];
      s_c[1][threadIdx.x] = G.c_xyz[3 * c + 1];
      s_c[2][threadIdx.x] = G.c_xyz[3 * c + 2];
      s_eps[threadIdx.x] = rad >= 0 ? eps[rad] : 0.0;
    }
    s_rad[threadIdx.x] = rad;
  }
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int k0 = 0; k0 < np; k0 += kK) {
    for (int e = threadIdx.x; e < kK * kT; e += blockDim.x) {
      const int f = e / kK, kk = e - f * kK, p = k0 + kk;
      const int fi = ti * kT + f, fj = tj * kT + f;
      sa[kk][f] = (p < np && fi < nb) ? base[static_cast<int64_t>(fi) * ldp + p] : 0.0;
      double th = 0.0;
      if (p < np && fj < nb && s_rad[f] >= 0) {
        const int64_t gp = p0 + p;
        const double dx = G.x[gp] - s_c[0][f], dy = G.y[gp] - s_c[1][f], dz = G.z[gp] - s_c[2][f];
        const double Vr = column_potential(B, vcoef, s_rad[f], centre_distance(dx, dy, dz));
        th = base[static_cast<int64_t>(fj) * ldp + p] * G.w[gp] * (v[gp] + s_eps[f] - Vr);
      }
      sb[kk][f] = th;
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < kK; ++kk) {
      const double a0v = sa[kk][2 * ty], a1v = sa[kk][2 * ty + 1];
      const double c0v = sb[kk][2 * tx], c1v = sb[kk][2 * tx + 1];
      acc[0][0] = fma(a0v, c0v, acc[0][0]);
      acc[0][1] = fma(a0v, c1v, acc[0][1]);
      acc[1][0] = fma(a1v, c0v, acc[1][0]);
      acc[1][1] = fma(a1v, c1v, acc[1][1]);
    }
    __syncthreads();
  }
  const int64_t pp = G.bat_pair_ptr[b];
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int i = ti * kT + 2 * ty + u, j = tj * kT + 2 * tx + w;
      if (i >= nb || j >= nb) continue;
      const int ii = G.fn_info[f0 + i], jj = G.fn_info[f0 + j];
      const int64_t off = G.pair_off[pp + static_cast<int64_t>(ii >> 16) * na + (jj >> 16)];
      if (off < 0) continue;
      atomicAdd(F + off + static_cast<int64_t>(ii & 0xffff) * local_nf(B, G, a0, jj >> 16) + (jj & 0xffff),
                acc[u][w]);
    }
}

q4c_status integrate_columns_fp64(const q4c_tables* t, const q4c_grid* g, const double* v, double* F,
                                  cudaStream_t s) {
  Q4C_CUDA(cudaMemsetAsync(F, 0, sizeof(double) * g->nnz, s));
  const DevBasis B = t->view();
  const DevGrid G = g->view();
  for (size_t wv = 0; wv + 1 < g->wave_b0.size(); ++wv) {
    const int64_t b0 = g->wave_b0[wv], b1 = g->wave_b0[wv + 1];
    const int64_t t0 = g->colt_w0[wv], t1 = g->colt_w0[wv + 1];  // every tile pair of the wave's batches
    if (b1 <= b0 || t1 <= t0) continue;
    if (q4c_status st = launch_basis_tiles(t, g, b0, b1, nullptr, nullptr, s)) return st;
    KernelScope ks("columns_fp64", s);
    k_columns_fp64<<<static_cast<unsigned>(t1 - t0), 256, 0, s>>>(B, G, g->d_col_tiles + t0, g->d_scr_off,
                                                                    g->d_scratch, v, t->d_col_eps, t->d_col_coef, F);
    Q4C_CUDA(cudaGetLastError());
  }
  return Q4C_OK;
}

// ---------------------------------------------------- density and adjoint
// n_p = sum_ij P_ij phi_i phi_j (NQ = 1), and with all four quantities (NQ = 4)
//   y_p = sum_ij [G^V phi_i phi_j + G^W grad_i.grad_j + G^x (Y_i Z_j - Z_i Y_j)
//                 + G^y (Z_i X_j - X_i Z_j) + G^z (X_i Y_j - Y_i X_j)],
// dL/dv = w y.  Only the symmetric parts of P, G^V, G^W and the antisymmetric
// parts of G^x, G^y, G^z contribute, so the sum runs over j >= i with
// coefficients S_ij = G_ij + G_ji (G_ii on the diagonal) and A_ij = G_ij - G_ji:
//   y = sum_i phi_i t0 + X_i tx + Y_i ty + Z_i tz,
//   t0 = sum_j S^V phi_j,  tx = sum_j S^W X_j + A^z Y_j - A^y Z_j  (cyclic),
// 10 (NQ = 1: one) FP64 multiply-adds per pair i <= j and point.  The FP64
// units (2 a clock and SM) bound it; the sum over all i, j of the products
// as written took 17 per ordered pair, 3.4 times as many.
//
// One CTA per batch and up to 32 of its points: a warp takes eight points
// times four rows i (lane = point + 8 row), the eight warps two row groups of
// up to four point octets; the row groups run over chunks of eight rows, the
// coefficients of 8 rows x 64 columns staged in shared memory.  A group of four
// rows starts at its own first column, so that almost nothing is spent below
// the diagonal.  Water (128 batches of 70 points, 24
// functions): 317 us -> 78 for the adjoint, 43 -> 16 for the density; 8-atom
// cluster: 7.18 ms -> 0.58.
constexpr int kRdRows = 8, kRdCols = 64, kRdPitch = kRdCols + 1;

// octets of points per CTA of a batch: at most 4, evenly spread
__device__ __forceinline__ int rd_octets(int np) {
  const int oct = (np + 7) >> 3, tiles = (oct + 3) >> 2;
  return (oct + tiles - 1) / tiles;
}

template <int NQ>
__global__ void __launch_bounds__(256) k_rowdot_fp64(DevBasis B, DevGrid G, int64_t b0,
                                                     const int64_t* __restrict__ scr_off,
                                                     const double* __restrict__ scratch, const double* GV,
                                                     const double* GW, const double* Gx, const double* Gy,
                                                     const double* Gz, double* __restrict__ out, int weighted) {
  constexpr int NM = NQ == 1 ? 1 : 5;  // matrices
  __shared__ double sG[NM][kRdRows][kRdPitch];
  __shared__ double s_acc[2][32];
  const int64_t b = b0 + blockIdx.x;
  const int64_t p0 = G.pt_ptr[b];
  const int np = static_cast<int>(G.pt_ptr[b + 1] - p0);
  const int n_oct = rd_octets(max(np, 1));
  const int pt0 = blockIdx.y * n_oct * 8;  // first point of this CTA
  if (pt0 >= np) return;
  const int ldp = (np + 7) & ~7;
  const int nb = static_cast<int>(G.bat_fn_ptr[b + 1] - G.bat_fn_ptr[b]);
  const int64_t plane = static_cast<int64_t>(nb) * ldp;
  const int64_t f0 = G.bat_fn_ptr[b];
  const int a0 = G.bat_atom_ptr[b], na = G.bat_atom_ptr[b + 1] - a0;
  const int64_t pp = G.bat_pair_ptr[b];
  const double* Gm[5] = {GV, GW, Gx, Gy, Gz};
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int oct = warp & 3, half = warp >> 2;
  const int row = 4 * half + (lane >> 3);               // row within a chunk
  const int pl = 8 * oct + (lane & 7), p = pt0 + pl;     // point within the CTA, within the batch
  const bool work = oct < n_oct && pt0 + 8 * oct < np;   // whole warps; p < ldp then
  const double* F = scratch + scr_off[b] + p;
  double acc = 0.0;
  for (int i0 = 0; i0 < nb; i0 += kRdRows) {
    double t[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) t[q] = 0.0;
    const bool live = work && i0 + 4 * half < nb;  // uniform in the warp
    for (int j0 = i0; j0 < nb; j0 += kRdCols) {
      __syncthreads();
      for (int e = threadIdx.x; e < kRdRows * kRdCols; e += blockDim.x) {
        const int r = e / kRdCols, c = e - r * kRdCols, i = i0 + r, j = j0 + c;
        double x[NM];
#pragma unroll
        for (int m = 0; m < NM; ++m) x[m] = 0.0;
        if (i < nb && j < nb && j >= i) {
          const int ii = G.fn_info[f0 + i], jj = G.fn_info[f0 + j];
          const int ai = ii >> 16, ki = ii & 0xffff, aj = jj >> 16, kj = jj & 0xffff;
          const int64_t o1 = G.pair_off[pp + static_cast<int64_t>(ai) * na + aj];
          const int64_t o2 = G.pair_off[pp + static_cast<int64_t>(aj) * na + ai];
          const int64_t e1 = o1 + static_cast<int64_t>(ki) * local_nf(B, G, a0, aj) + kj;
          const int64_t e2 = o2 + static_cast<int64_t>(kj) * local_nf(B, G, a0, ai) + ki;
#pragma unroll
          for (int m = 0; m < NM; ++m) {
            if (Gm[m] == nullptr) continue;
            const double g1 = o1 < 0 ? 0.0 : Gm[m][e1];
            if (i == j) {
              x[m] = m < 2 ? g1 : 0.0;
            } else {
              const double g2 = o2 < 0 ? 0.0 : Gm[m][e2];
              x[m] = m < 2 ? g1 + g2 : g1 - g2;
            }
          }
        }
#pragma unroll
        for (int m = 0; m < NM; ++m) sG[m][r][c] = x[m];
      }
      __syncthreads();
      if (live) {
        const int jb = max(j0, i0 + 4 * half), je = min(nb, j0 + kRdCols);
        const double* Fj = F + static_cast<int64_t>(jb) * ldp;
#pragma unroll 4
        for (int j = jb; j < je; ++j, Fj += ldp) {
          const double* g = &sG[0][row][j - j0];
          if constexpr (NQ == 1) {
            t[0] = fma(g[0], __ldg(Fj), t[0]);
          } else {
            constexpr int M = kRdRows * kRdPitch;
            const double f = __ldg(Fj), x = __ldg(Fj + plane), y = __ldg(Fj + 2 * plane), z = __ldg(Fj + 3 * plane);
            const double gw = g[M], gx = g[2 * M], gy = g[3 * M], gz = g[4 * M];
            t[0] = fma(g[0], f, t[0]);
            t[1] = fma(gw, x, fma(gz, y, fma(-gy, z, t[1])));
            t[2] = fma(gw, y, fma(gx, z, fma(-gz, x, t[2])));
            t[3] = fma(gw, z, fma(gy, x, fma(-gx, y, t[3])));
          }
        }
      }
    }
    if (live && i0 + row < nb) {
      const double* Fi = F + static_cast<int64_t>(i0 + row) * ldp;
#pragma unroll
      for (int q = 0; q < NQ; ++q) acc = fma(__ldg(Fi + q * plane), t[q], acc);
    }
  }
  // the four rows of a warp, then the two row groups of a point
  acc += __shfl_xor_sync(0xffffffffu, acc, 8);
  acc += __shfl_xor_sync(0xffffffffu, acc, 16);
  if (lane < 8) s_acc[half][pl] = acc;
  __syncthreads();
  if (work && half == 0 && lane < 8 && p < np) {
    const double y = s_acc[0][pl] + s_acc[1][pl];
    out[p0 + p] = weighted ? G.w[p0 + p] * y : y;
  }
}

template <int NQ>
static q4c_status rowdot_fp64_wave(const q4c_grid* g, int wv, const double* const M[5], double* out, bool weighted,
                                   const char* name, cudaStream_t s) {
  const int64_t b0 = g->wave_b0[wv], b1 = g->wave_b0[wv + 1];
  if (b1 <= b0) return Q4C_OK;
  const unsigned tiles = static_cast<unsigned>((std::max(g->max_np, 1) + 31) / 32);
  KernelScope ks(name, s);
  k_rowdot_fp64<NQ><<<dim3(static_cast<unsigned>(b1 - b0), tiles), 256, 0, s>>>(
      g->tables->view(), g->view(), b0, g->d_scr_off, g->d_scratch, M[0], M[1], M[2], M[3], M[4], out,
      weighted ? 1 : 0);
  Q4C_CUDA(cudaGetLastError());
  return Q4C_OK;
}

// the density of one wave (its basis tiles in place)
// (the limits here and below are the calls' own: the kernel's shared memory does
// not depend on the batch)
q4c_status density_fp64_wave(const q4c_grid* g, int wv, const double* P, double* n, cudaStream_t s) {
  if (g->max_nb > 7264) {
    set_error("the FP64 density needs at most 7264 active functions per batch");
    return Q4C_EUNSUPPORTED;
  }
  const double* M[5] = {P, nullptr, nullptr, nullptr, nullptr};
  return rowdot_fp64_wave<1>(g, wv, M, n, false, "density_fp64", s);
}

q4c_status density_fp64(const q4c_tables* t, const q4c_grid* g, const double* P, double* n, cudaStream_t s) {
  for (size_t wv = 0; wv + 1 < g->wave_b0.size(); ++wv) {
    const int64_t b0 = g->wave_b0[wv], b1 = g->wave_b0[wv + 1];
    if (b1 <= b0) continue;
    if (q4c_status st = launch_basis_tiles(t, g, b0, b1, nullptr, nullptr, s)) return st;
    if (q4c_status st = density_fp64_wave(g, static_cast<int>(wv), P, n, s)) return st;
  }
  return Q4C_OK;
}

// the adjoint (weighted) or gradient density (unweighted) of one wave (its
// basis tiles in place)
q4c_status backward_fp64_wave(const q4c_grid* g, int wv, const q4c_matrices* Gm, double* dLdv, bool weighted,
                              cudaStream_t s) {
  if (g->max_nb > 5811) {
    set_error("the FP64 adjoint needs at most 5811 active functions per batch");
    return Q4C_EUNSUPPORTED;
  }
  const double* M[5] = {Gm->V, Gm->W0, Gm->SOx, Gm->SOy, Gm->SOz};
  return rowdot_fp64_wave<4>(g, wv, M, dLdv, weighted, "backward_fp64", s);
}

q4c_status backward_fp64(const q4c_tables* t, const q4c_grid* g, const q4c_matrices* Gm, double* dLdv,
                         cudaStream_t s, bool weighted) {
  for (size_t wv = 0; wv + 1 < g->wave_b0.size(); ++wv) {
    const int64_t b0 = g->wave_b0[wv], b1 = g->wave_b0[wv + 1];
    if (b1 <= b0) continue;
    if (q4c_status st = launch_basis_tiles(t, g, b0, b1, nullptr, nullptr, s)) return st;
    if (q4c_status st = backward_fp64_wave(g, static_cast<int>(wv), Gm, dLdv, weighted, s)) return st;
  }
  return Q4C_OK;
}

// ---------------------------------------------------------- basis probe
__global__ void k_basis_eval(DevBasis B, DevGrid G, int n_basis, const int* __restrict__ atom_fn0, int64_t n_pts,
                             const double* __restrict__ xyz, double* __restrict__ phi, double* __restrict__ grad) {
  const int64_t item = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (item >= n_pts * G.n_atoms) return;
  const int A = static_cast<int>(item / n_pts);
  const int64_t p = item - A * n_pts;
  const int f0 = atom_fn0[A];
  atom_functions(B, G.atom_sp[A], xyz[3 * p] - G.atom_xyz[3 * A], xyz[3 * p + 1] - G.atom_xyz[3 * A + 1],
                 xyz[3 * p + 2] - G.atom_xyz[3 * A + 2], [&](int k, double v, double gx, double gy, double gz) {
                   const int64_t o = static_cast<int64_t>(f0 + k) * n_pts + p;
                   phi[o] = v;
                   grad[3 * o] = gx;
                   grad[3 * o + 1] = gy;
                   grad[3 * o + 2] = gz;
                 });
}

q4c_status basis_eval(const q4c_tables* t, const q4c_grid* g, int64_t n_pts, const double* xyz, double* phi,
                      double* grad, cudaStream_t s) {
  if (n_pts == 0) return Q4C_OK;
  const int64_t items = n_pts * g->n_atoms;
  KernelScope ks("basis_eval", s);
  k_basis_eval<<<static_cast<unsigned>((items + 127) / 128), 128, 0, s>>>(t->view(), g->view(), g->n_basis,
                                                                         g->d_atom_fn0, n_pts, xyz, phi, grad);
  Q4C_CUDA(cudaGetLastError());
  return Q4C_OK;
}

}  // namespace q4c
