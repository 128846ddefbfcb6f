// Split-precision batch products for batches of more than 256 functions: two
// 64-function row tiles per step against one B operand.
//
// The slices, their levels and the outputs are those of split.cu.  An accumulator
// of at most 341 terms (points times the products that share it) takes digits one
// bit finer: |d_0| <= 128, resolving 2^-47 of the column's largest value, with
// levels 0-2 sums of at most 2^14, 2^15 and 3 2^14 units per term, exact.  A longer
// one keeps split.cu's |d_0| <= 64: level 1 is then exact for every batch (2^14
// units a term, at most 1,023 terms) and level 2 for 512 terms, beyond which a
// rounding of L2 sits ~2^-40 below the column scale.  With the finer digits there
// level 1 itself would pass 2^24 and lose its last bits ~2^-32 below the column
// scale: W0 of 340 points with digits of one sign 1e-9 off, 1e-15 so.
//
// Layout: M = 128 rows are two halves of 64 functions with a product each, both
// against the same B operand: two row tiles of one output, or two outputs of
// one tile.  The A digits live in tensor memory (the slicers write them there,
// 8 columns a digit), the B digits B_0 .. B_5 back to back in shared memory, so
// that A_s times [B_0 .. B_(5-s)] is one MMA of N = w (6 - s) columns (two where
// that is above 256) that adds levels s .. 5 to consecutive blocks of w columns:
// the twenty-one slice pairs with s + t <= 5 of both halves in six to eight MMAs.
//
// Row tiles ti <= tj go in pairs: V, W0 (three products into one accumulator,
// sliced against a common exponent per function) and SO_x = (D Y)^T Z - (D Z)^T Y
// etc. (two products).  A last single one is the diagonal tile, whose SO come
// from A_yz = (D Y)^T Z etc. alone (SO_x = A_yz - A_yz^T, applied while
// scattering), one beside V, two beside each other, each step's B operand sliced
// against its own exponents; its W0 runs alone.  The per-column operator is Phi
// against Psi on every tile pair.
//
// What bounds it: slicing.  A step of two products slices 192 rows of 16 values
// (about 630 issue slots a scheduler) where two steps of split.cu slice 256, and its
// MMAs read 43 KB from shared memory where theirs read 97.  Measured per 64 x 64
// x 16 product: 710 clocks for 1,185 on batches of 700 functions (304-atom slab,
// products 44.0 -> 33.7 ms); with few row tiles half of M is empty much of the
// time and split.cu is the faster one (64-atom cluster, 65-128 functions: 2.15 ms
// there, 3.2 here; 129-205: 0.59 and 0.74).
#include <cuda.h>

#include <algorithm>

#include "internal.h"
#include "tc.cuh"

namespace q4c {
namespace pairs {
using namespace tc;

constexpr int kTile = 64;                    // functions per tile (one half of M)
constexpr int kKc = 16;                      // points per step (one K = 16 MMA step)
constexpr int kSBO = (kKc / 8) * 128;        // 256 B between 8-row groups
constexpr int kASlicers = 256;               // warps 0-7 slice the A operand
constexpr int kBWarp0 = 8;                   // warps 8-11 slice the B operand
constexpr int kBSlicers = 128;
constexpr int kEpiWarp0 = 12;                // warps 12-19 drain tensor memory (two groups of four)
constexpr int kEpiThreads = 256;
constexpr int kMmaWarp = 20;                 // warp 20 owns tensor memory and issues the MMAs
constexpr int kProdWarp = 21;                // warp 21 issues the TMA loads of the raw operands
constexpr int kThreads = 22 * 32;
constexpr int kStageB = kSlices * kTile * kRowBytes;  // [B0..B5] of one step, 12 KB
constexpr int kStagesB = 4;
constexpr int kRawTile = kTile * kKc * 8;            // one 64 x 16 box of (hi, lo), 8 KB
constexpr int kRawStep = 3 * kRawTile + 1024;        // A top, A bottom and B boxes, the step's D values; 1024-aligned
constexpr int kEpiPitch = kTile + 1;                 // (hi, lo) pairs per staged row
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kTmemA = 384;  // two stages of six A digits (48 columns) behind six levels of up to 64

// Shared memory: four raw stages of one step (two of two steps, half the handshakes,
// are the slower by far: 304-atom slab 54.2 ms for 33.7), the B digits, the staged
// elements.
constexpr int kRaw = 4;
constexpr int kSmemB = kRaw * kRawStep;
constexpr int kSmemEpi = kSmemB + kStagesB * kStageB;  // [128][kEpiPitch] pairs
constexpr int kSmemBar = kSmemEpi + 2 * kTile * kEpiPitch * 8;
// raw full/empty, B full/empty, A full[2], A empty[2], acc full, acc empty, drain
constexpr int kNumBars = 2 * kRaw + 2 * kStagesB + 7;
constexpr int kSmemTotal = kSmemBar + kNumBars * 8 + 16;
static_assert(kSmemTotal <= 232448, "shared memory per CTA");

// ------------------------------------------------------------ items
// An item is (batch, type, B tile tj, row tiles ti0 | ti1 << 16); ti1 = 0xffff: no
// bottom half.  Its program is up to three products K-concatenated step by step:
// per product the B quantity and for each half the A quantity (0 Phi, 1 X, 2 Y,
// 3 Z; + 4: subtracted, D negated; + 8: present).
// kDiagV, kDiagA: the halves are different outputs of a diagonal tile, a step each.
enum Type { kV = 0, kW0 = 1, kSOx = 2, kSOy = 3, kSOz = 4, kCol = 5, kDiagV = 6, kDiagA = 7 };
struct Step {
  int b, top, bot;
};
constexpr unsigned step_code(int b, int top, int bot) { return static_cast<unsigned>(b | top << 2 | bot << 6); }
constexpr unsigned program(unsigned s0, unsigned s1 = 0, unsigned s2 = 0) { return s0 | s1 << 10 | s2 << 20; }
__device__ __forceinline__ int n_products(int type) {
  return static_cast<int>((0x22122231u >> (4 * type)) & 15u);  // types 7 .. 0
}
__device__ __forceinline__ Step step_of(int type, int s) {
  unsigned p;
  switch (type) {
    case kV: p = program(step_code(0, 8, 8)); break;
    case kW0: p = program(step_code(1, 9, 9), step_code(2, 10, 10), step_code(3, 11, 11)); break;
    case kSOx: p = program(step_code(3, 10, 10), step_code(2, 15, 15)); break;  // Y Z - Z Y
    case kSOy: p = program(step_code(1, 11, 11), step_code(3, 13, 13)); break;  // Z X - X Z
    case kSOz: p = program(step_code(2, 9, 9), step_code(1, 14, 14)); break;    // X Y - Y X
    case kCol: p = program(step_code(1, 8, 8)); break;                          // Phi Psi
    case kDiagV: p = program(step_code(1, 11, 0), step_code(0, 0, 8)); break;   // A_zx; V
    default: p = program(step_code(2, 9, 0), step_code(3, 0, 10)); break;       // A_xy; A_yz
  }
  p >>= 10 * s;
  return {static_cast<int>(p & 3u), static_cast<int>((p >> 2) & 15u), static_cast<int>((p >> 6) & 15u)};
}
// bits by which the digits of an item of n_p points are finer than tc::slice6x2's
// against the exponent itself: one where the terms of an accumulator stay at 341
__device__ __forceinline__ int fine_of(int type, int np) {
  const int k = type == kW0 ? 3 : type >= kSOx && type <= kSOz ? 2 : 1;  // products in an accumulator
  return k * np <= 341 ? 1 : 0;
}
// output of a half: 0 V (or F), 1 W0, 2-4 SO
__device__ __forceinline__ int output_of(int type, bool bot) {
  return type <= kSOz ? type : type == kCol ? 0 : type == kDiagV ? (bot ? 0 : 3) : (bot ? 2 : 4);
}

// B-tile width of an item: the functions of tile tj rounded up to 16 (the
// MMA's N granularity)
__device__ __forceinline__ int item_w(int nb, int tj) { return (min(kTile, nb - tj * kTile) + 15) & ~15; }

__device__ __forceinline__ float4 lds128(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}

__device__ __forceinline__ void sts128(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}

// four tensor-memory columns of this warp's lanes
__device__ __forceinline__ void tmem_st4(uint32_t t, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(t), "r"(x), "r"(y), "r"(z), "r"(w)
               : "memory");
}

// A from tensor memory, B from shared memory
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(d),
      "r"(a), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

// The 21 slice products of one step: A digit s (8 columns at a + 8 s) times
// [B_0 .. B_(5-s)] (w rows of 32 B each) into levels s .. 5 (w columns each)
__device__ __forceinline__ void mma_step(uint32_t d, uint32_t a, uint64_t b, int w, bool first, uint32_t neg) {
#pragma unroll
  for (int s = 0; s < kSlices; ++s) {
    const int n = w * (kSlices - s);
    const uint32_t acc = (first && s == 0) ? 0u : 1u;
    mma_ts(d + s * w, a + 8 * s, b, make_idesc(128, min(n, 256)) | neg, acc);
    if (s < 2 && n > 256)
      mma_ts(d + s * w + 256, a + 8 * s, b + (256 * kRowBytes >> 4), make_idesc(128, n - 256) | neg, acc);
  }
}

// One work item; its K dimension is a stream of steps of 16 points, the
// item's products interleaved step by step.
//
// Warp roles (one CTA per SM, items strided over the CTAs):
//   warp 21     (one thread) loads step g's raw operands once the slicers have
//               read the stage (raw_empty): TMA boxes of the A rows of the halves
//               that take part and of the B rows (zeros past n_p and n_b) and the
//               step's 16 D values; one mbarrier (raw_full) counts the bytes;
//   warps 0-7   thread (row of M, points 8h .. 8h + 7) forms the D-scaled values
//               in double-float, slices them and writes the six digits to tensor
//               memory stage g mod 2 once the MMAs that last read it have
//               completed (a_empty, a tcgen05.commit), then arrives on a_full;
//   warps 8-11  thread (row of B, points 8h .. 8h + 7) slices into operand stage
//               g mod 4 (b_empty, b_full);
//   warp 20     waits for both operands, issues the step's MMAs, commits a_empty
//               and b_empty, and after an item's last step acc_full;
//   warps 12-19 wait acc_full, combine the six levels of every element into an FP32
//               pair in shared memory, hand the accumulators back (acc_empty) and
//               scatter while the next item runs.
// Every wait is bounded; a role that times out sets the status bit and an
// abort flag that ends the other roles' waits, and the MMA warp drains its
// outstanding MMAs (bounded) before tensor memory is freed.
__global__ void __launch_bounds__(kThreads, 1)
    k_split_pairs(DevGrid G, const int4* __restrict__ items, int n_items, const CUtensorMap* __restrict__ maps,
                  const float2* __restrict__ dpad, const int* __restrict__ colexp, double* V, double* W0, double* SOx,
                  double* SOy, double* SOz, unsigned* status) {
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kSmemBar);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kSmemBar + kNumBars * 8);
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + kSmemBar + kNumBars * 8 + 4);

  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  const uint32_t smem0 = smem_u32(smem);
  if (smem0 & 1023u) {  // the swizzled TMA boxes need 1024-byte aligned stages
    if (tid == 0) atomicOr(status, 2u);
    return;
  }
  const uint32_t bar0 = smem_u32(bars);
  auto rawfull_bar = [&](int k) { return bar0 + 8u * k; };
  auto rawempty_bar = [&](int k) { return bar0 + 8u * (kRaw + k); };
  auto bfull_bar = [&](int k) { return bar0 + 8u * (2 * kRaw + k); };
  auto bempty_bar = [&](int k) { return bar0 + 8u * (2 * kRaw + kStagesB + k); };
  auto afull_bar = [&](int k) { return bar0 + 8u * (2 * kRaw + 2 * kStagesB + k); };
  auto aempty_bar = [&](int k) { return bar0 + 8u * (2 * kRaw + 2 * kStagesB + 2 + k); };
  const uint32_t accfull_bar = bar0 + 8u * (2 * kRaw + 2 * kStagesB + 4);
  const uint32_t accempty_bar = bar0 + 8u * (2 * kRaw + 2 * kStagesB + 5);
  const uint32_t drain_bar = bar0 + 8u * (2 * kRaw + 2 * kStagesB + 6);

  if (tid == 0) {
    for (int k = 0; k < kRaw; ++k) {
      mbar_init(rawfull_bar(k), 1);
      mbar_init(rawempty_bar(k), (kASlicers / 2 + kBSlicers) / 32);  // an A group, the B warps
    }
    for (int k = 0; k < kStagesB; ++k) {
      mbar_init(bfull_bar(k), kBSlicers);
      mbar_init(bempty_bar(k), 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(afull_bar(k), kASlicers / 2);
      mbar_init(aempty_bar(k), 1);
    }
    mbar_init(accfull_bar, 1);
    mbar_init(accempty_bar, kEpiThreads);
    mbar_init(drain_bar, 1);
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
  // steps of an item: each chunk of 16 points once per product
  auto item_np = [&](const int4& it) { return static_cast<int>(G.pt_ptr[it.x + 1] - G.pt_ptr[it.x]); };
  auto item_steps = [&](const int4& it) { return (item_np(it) + kKc - 1) / kKc * n_products(it.y); };

  if (warp < kBWarp0) {
    // ---------------------------------------------------------- A slicers
    // thread = tensor-memory lane 32 (warp & 3) + lane (row of M) and the step's 16
    // points; a group of four warps takes every other step and owns one stage
    const int ag = warp >> 2;
    const int row = (warp & 3) * 32 + lane;
    const bool bot = row >= kTile;  // uniform in the warp
    const int r64 = row & (kTile - 1);
    // raw box row r64 is 128 bytes, its 16-byte chunk c swizzled to c ^ (r & 7)
    const uint32_t box = (bot ? kRawTile : 0) + r64 * 128;
    const uint32_t t = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + kTmemA + ag * 48;
    int g = 0, aph = 1;  // steps, parity
    bool ok = true;
    for (int n = blockIdx.x; n < n_items && ok; n += gridDim.x) {
      const int4 item = items[n];
      const int type = item.y, n_prod = n_products(type);
      const int64_t fn0 = G.bat_fn_ptr[item.x];
      const int nb = static_cast<int>(G.bat_fn_ptr[item.x + 1] - fn0);
      const int n_st = item_steps(item);
      const int ti = bot ? static_cast<int>(static_cast<unsigned>(item.w) >> 16) : item.w & 0xffff;
      // rounding constant of this row: products that share an accumulator are
      // sliced against one exponent per function; acts: products that take part
      int e = -30000;
      unsigned acts = 0;
      for (int s = 0; s < n_prod && ti != 0xffff; ++s) {
        const Step st = step_of(type, s);
        const int a = bot ? st.bot : st.top;
        if (!(a & 8)) continue;
        acts |= 1u << s;
        if (ti * kTile + r64 < nb) e = max(e, __ldg(colexp + 8 * fn0 + (a & 3) * nb + ti * kTile + r64));
      }
      const float mag = magic0(e - fine_of(type, item_np(item)));
      const float mm[4] = {mag, mag, mag, mag};
      for (int s = 0, pr = 0; s < n_st && ok; ++s, ++g, pr = pr + 1 == n_prod ? 0 : pr + 1) {
        const bool act = acts >> pr & 1u;
        const int rs = g % kRaw;
        if ((g & 1) != ag) continue;
        if (!mbar_wait_warp(rawfull_bar(rs), (g / kRaw) & 1, s_abort, status, G.wait_ns)) {
          ok = false;
          break;
        }
        const uint32_t raw = smem0 + rs * kRawStep;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          uint32_t wd[4][kSlices];
          if (act) {
            float2 x[4], l[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {  // points 8 half + 2u, + 1: D-scaled values in double-float
              const float4 v = lds128(raw + box + (((4 * half + u) ^ (r64 & 7)) << 4));
              const float4 d = lds128(raw + 3 * kRawTile + (4 * half + u) * 16);
              df_mul2(pk2(v.x, v.z), pk2(v.y, v.w), pk2(d.x, d.z), pk2(d.y, d.w), pk2(-d.x, -d.z), x[u], l[u]);
            }
            slice_pairs<4>(x, l, mm, wd);
          } else {
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
              for (int d = 0; d < kSlices; ++d) wd[u][d] = 0u;
          }
          if (half == 0) {  // the first half is sliced while the stage's last MMAs still run
            if (!mbar_wait_warp(aempty_bar(ag), aph, s_abort, status, G.wait_ns)) {
              ok = false;
              break;
            }
            tc_fence_after();
          }
#pragma unroll
          for (int d = 0; d < kSlices; ++d)
            tmem_st4(t + 8 * d + 4 * half, wd[0][d], wd[1][d], wd[2][d], wd[3][d]);
        }
        if (!ok) break;
        aph ^= 1;
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before();
        mbar_arrive(afull_bar(ag));
        // The raw stage is free: the digits above were formed from its values,
        // so the loads have landed.
        __syncwarp();
        if (lane == 0) mbar_arrive(rawempty_bar(rs));
      }
    }
  } else if (warp < kBWarp0 + kBSlicers / 32) {
    // ---------------------------------------------------------- B slicers
    // row 32 (warp & 1) + lane of the B tile, points 8 half .. 8 half + 7
    const int half = (warp >> 1) & 1, r64 = (warp & 1) * 32 + lane;
    const uint32_t box = 2 * kRawTile + r64 * 128;
    const uint32_t dstB = (r64 >> 3) * kSBO + half * kLBO + (r64 & 7) * 16;
    int g = 0;
    bool ok = true;
    for (int n = blockIdx.x; n < n_items && ok; n += gridDim.x) {
      const int4 item = items[n];
      const int type = item.y, n_prod = n_products(type);
      const int64_t fn0 = G.bat_fn_ptr[item.x];
      const int nb = static_cast<int>(G.bat_fn_ptr[item.x + 1] - fn0);
      const int n_st = item_steps(item);
      const int w = item_w(nb, item.z);
      const bool have = r64 < w;
      int e = -30000, e1 = -30000;
      for (int s = 0; s < n_prod; ++s) {
        const int f = item.z * kTile + r64;
        if (f >= nb) break;
        const int v = __ldg(colexp + 8 * fn0 + (4 + step_of(type, s).b) * nb + f);
        if (type >= kDiagV && s == 1)
          e1 = v;  // its two products go to different accumulators
        else
          e = max(e, v);
      }
      const int fine = fine_of(type, item_np(item));
      const float mag = magic0(e - fine), mag1 = type >= kDiagV ? magic0(e1 - fine) : mag;
      for (int s = 0, pr = 0; s < n_st; ++s, ++g, pr = pr + 1 == n_prod ? 0 : pr + 1) {
        const int rs = g % kRaw;
        if (!mbar_wait_warp(rawfull_bar(rs), (g / kRaw) & 1, s_abort, status, G.wait_ns)) {
          ok = false;
          break;
        }
        const float m = pr ? mag1 : mag;
        const float mm[4] = {m, m, m, m};
        const uint32_t raw = smem0 + rs * kRawStep;
        uint32_t wd[4][kSlices];
        if (have) {
          float2 x[4], l[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 v = lds128(raw + box + (((4 * half + u) ^ (r64 & 7)) << 4));
            x[u] = pk2(v.x, v.z);
            l[u] = pk2(v.y, v.w);
          }
          slice_pairs<4>(x, l, mm, wd);
        }
        const int st = g % kStagesB;
        if (!mbar_wait_warp(bempty_bar(st), ((g / kStagesB) & 1) ^ 1, s_abort, status, G.wait_ns)) {
          ok = false;
          break;
        }
        if (have) {
          const uint32_t dst = smem0 + kSmemB + st * kStageB + dstB;
#pragma unroll
          for (int d = 0; d < kSlices; ++d) sts128(dst + d * w * kRowBytes, wd[0][d], wd[1][d], wd[2][d], wd[3][d]);
        }
        fence_async_smem();
        mbar_arrive(bfull_bar(st));
        __syncwarp();
        if (lane == 0) mbar_arrive(rawempty_bar(rs));
      }
    }
  } else if (warp == kProdWarp) {
    // ---------------------------------------------------------- TMA producer
    if (lane == 0) {
      int rs = 0, ph = 1, g = 0;
      bool ok = true;
      for (int n = blockIdx.x; n < n_items && ok; n += gridDim.x) {
        const int4 item = items[n];
        const int n_st = item_steps(item), n_prod = n_products(item.y);
        const CUtensorMap* map = maps + item.x;
        const float2* drow = dpad + static_cast<int64_t>(item.x) * kDPitch;
        const int ti1 = static_cast<int>(static_cast<unsigned>(item.w) >> 16);
        const int i0 = (item.w & 0xffff) * kTile, i1 = ti1 * kTile, j0 = item.z * kTile;
        for (int s = 0, pr = 0, c = 0; s < n_st; ++s, ++g) {
          if (!mbar_wait_abort(rawempty_bar(rs), ph, s_abort, status, G.wait_ns)) {
            ok = false;
            break;
          }
          const Step stp = step_of(item.y, pr);
          const bool top = stp.top & 8, bot = (stp.bot & 8) && ti1 != 0xffff;
          const uint32_t fb = rawfull_bar(rs);
          arrive_expect_tx(fb, (1 + top + bot) * kRawTile + kKc * 8);
          const uint32_t dst = smem0 + rs * kRawStep;
          const int x = c * kKc;  // first point of the step (16-byte aligned coordinate)
          if (top) tma_load_3d(dst, map, x, i0, stp.top & 3, fb);
          if (bot) tma_load_3d(dst + kRawTile, map, x, i1, stp.bot & 3, fb);
          tma_load_3d(dst + 2 * kRawTile, map, x, j0, stp.b, fb);
          bulk_copy(dst + 3 * kRawTile, drow + x, kKc * 8, fb);
          if (++rs == kRaw) {
            rs = 0;
            ph ^= 1;
          }
          if (++pr == n_prod) {
            pr = 0;
            ++c;
          }
        }
      }
      // no copy outlives the CTA: the last kRaw issued stages have landed
      // (immediately true unless a wait gave up; bounded either way)
      for (int h = max(0, g - kRaw); h < g; ++h) (void)mbar_wait(rawfull_bar(h % kRaw), (h / kRaw) & 1, status);
    }
    __syncwarp();
  } else if (warp == kMmaWarp) {
    // ---------------------------------------------------------- MMA issue
    // (the whole warp waits, one lane issues, operands uniform: see rowdot.cu)
    int g = 0, k = 0;
    bool ok = true;
    const uint64_t descB = make_desc(smem0 + kSmemB, kSBO);
    for (int n = blockIdx.x; n < n_items && ok; n += gridDim.x, ++k) {
      const int4 item = items[n];
      const int n_steps = uniform(item_steps(item));
      const int w = uniform(item_w(static_cast<int>(G.bat_fn_ptr[item.x + 1] - G.bat_fn_ptr[item.x]), item.z));
      if (!mbar_wait_warp(accempty_bar, (k & 1) ^ 1, s_abort, status, G.wait_ns)) break;
      const int type = item.y, n_prod = n_products(type);
      for (int s = 0, pr = 0; s < n_steps; ++s, ++g) {
        // a subtracted product (both halves alike): the instruction's negate-A bit
        const uint32_t neg = (step_of(type, pr).top & 4) ? 1u << 13 : 0u;
        if (++pr == n_prod) pr = 0;
        const int sa = uniform(g & 1), sb = uniform(g % kStagesB);
        if (!mbar_wait_warp(bfull_bar(sb), (g / kStagesB) & 1, s_abort, status, G.wait_ns) ||
            !mbar_wait_warp(afull_bar(sa), (g >> 1) & 1, s_abort, status, G.wait_ns)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t b = descB + static_cast<uint32_t>(sb * (kStageB >> 4));
        if (elect_one()) {
          mma_step(tmem, tmem + kTmemA + sa * 48, b, w, s == 0, neg);
          mma_commit(aempty_bar(sa));
          mma_commit(bempty_bar(sb));
        }
      }
      if (ok && elect_one()) mma_commit(accfull_bar);
    }
    // every MMA issued by this warp has completed before tensor memory is freed
    if (elect_one()) {
      mma_commit(drain_bar);
      (void)mbar_wait(drain_bar, 0, status);
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------- epilogue
    const int eg = (warp - kEpiWarp0) >> 2;  // column group
    const int quarter = warp & 3;            // TMEM lanes 32 quarter .. +31
    const int r = quarter * 32 + lane;
    const int et = tid - kEpiWarp0 * 32;
    const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
    float2* stg = reinterpret_cast<float2*>(smem + kSmemEpi);
    int k = 0;
    for (int n = blockIdx.x; n < n_items; n += gridDim.x, ++k) {
      const int4 item = items[n];
      const int64_t b = item.x;
      const int nb = static_cast<int>(G.bat_fn_ptr[b + 1] - G.bat_fn_ptr[b]);
      const int w = item_w(nb, item.z);  // accumulator levels are w columns wide
      const int ti0 = item.w & 0xffff, ti1 = static_cast<int>(static_cast<unsigned>(item.w) >> 16);
      const int* idx = G.bat_idx + G.bat_idx_ptr[b];
      const bool ok = mbar_wait_warp(accfull_bar, k & 1, s_abort, status, G.wait_ns);
      if (bar_red_or(2, kEpiThreads, !ok)) break;  // also: the last item's pairs have been read
      tc_fence_after();
      if (quarter < 2 || ti1 != 0xffff) {
        for (int c = 8 * eg; c < w; c += 16) {
          float v[6][8];
          tmem_ld8x6(tmem + lane_base + c, w, v);
#pragma unroll
          for (int i = 0; i < 8; i += 2) {  // exact levels by two-sums, rounded tail on top
            float2 s, es, u, eu;
            two_sum2(pk2(v[0][i], v[0][i + 1]), pk2(v[1][i], v[1][i + 1]), s, es);
            two_sum2(s, pk2(v[2][i], v[2][i + 1]), u, eu);
            const float2 lo = add2(add2(es, eu), add2(pk2(v[3][i], v[3][i + 1]),
                                                      add2(pk2(v[4][i], v[4][i + 1]), pk2(v[5][i], v[5][i + 1]))));
            stg[r * kEpiPitch + c + i] = make_float2(u.x, lo.x);
            stg[r * kEpiPitch + c + i + 1] = make_float2(u.y, lo.y);
          }
        }
      }
      tc_fence_before();
      mbar_arrive(accempty_bar);
      bar_sync(2, kEpiThreads);
      // scatter: a warp covers 16 consecutive columns of two rows; eight
      // elements a thread at a time, their offsets loaded together
      const int col0 = et & 15, row0 = et >> 4;
      const int halves = ti1 != 0xffff ? 2 : 1, n_blk = (w >> 4) * halves;
      // block k: columns 16 (k / halves) .., half k % halves
      auto load_off = [&](int blk, int (&off)[4]) {
        const int hb = halves == 2 ? blk & 1 : 0, c0 = (halves == 2 ? blk >> 1 : blk) * 16;
        const int o = output_of(item.y, hb != 0);
        const bool sym = item.y != kCol && o <= 1, anti = item.y >= kDiagV && o >= 2;
        const int i0 = (hb ? ti1 : ti0) * kTile, j = item.z * kTile + c0 + col0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = i0 + row0 + 16 * q;
          // V and W0 where i <= j, SO where i < j; a diagonal tile's A_k gives
          // A_k(i, j) - A_k(j, i) at (i, j), i < j; the per-column operator all
          const bool swap = anti && i > j;
          const int ri = min(swap ? j : i, nb - 1), rj = min(swap ? i : j, nb - 1);
          const int v = __ldg(idx + ri * nb + rj);
          const bool use = i < nb && j < nb && (item.y == kCol || (sym ? i <= j : anti ? i != j : i < j));
          off[q] = use ? v : -1;
        }
      };
      int off[4], nxt[4];
      load_off(0, off);
      for (int blk = 0; blk < n_blk; ++blk) {
        if (blk + 1 < n_blk) load_off(blk + 1, nxt);  // a block ahead
        const int hb = halves == 2 ? blk & 1 : 0, c0 = (halves == 2 ? blk >> 1 : blk) * 16;
        const int o = output_of(item.y, hb != 0);
        const bool anti = item.y >= kDiagV && o >= 2;
        double* out = o == 0 ? V : o == 1 ? W0 : o == 2 ? SOx : o == 3 ? SOy : SOz;
        const int i0 = (hb ? ti1 : ti0) * kTile, j = item.z * kTile + c0 + col0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (off[q] >= 0) {
            const float2 x = stg[(hb * kTile + row0 + 16 * q) * kEpiPitch + c0 + col0];
            const bool neg = anti && i0 + row0 + 16 * q > j;
            atomicAdd(out + off[q], widen(neg ? -x.x : x.x) + widen(neg ? -x.y : x.y));
          }
          off[q] = nxt[q];
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

}  // namespace pairs

// one launch over items [0, n): a persistent grid of at most one CTA per SM
q4c_status launch_pairs(const q4c_grid* g, const int4* items, int n, double* V, double* W0, double* SOx, double* SOy,
                        double* SOz, const char* name, cudaStream_t s) {
  Q4C_CUDA(cudaFuncSetAttribute(pairs::k_split_pairs, cudaFuncAttributeMaxDynamicSharedMemorySize, pairs::kSmemTotal));
  int dev = 0, n_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  KernelScope ks(name, s);
  pairs::k_split_pairs<<<std::min(n, n_sm), pairs::kThreads, pairs::kSmemTotal, s>>>(
      g->view(), items, n, reinterpret_cast<const CUtensorMap*>(g->d_tmaps), g->d_dpad, g->d_colexp, V, W0, SOx, SOy,
      SOz, g->d_status);
  Q4C_CUDA(cudaGetLastError());
  return Q4C_OK;
}

}  // namespace q4c
