// umma32.cuh - an FP32 matrix product on the fifth-generation tensor cores,
// with the tree's element-wise remainder evaluated in its epilogue.
//
// The tensor cores multiply 16-bit operands; FP32 operands run there as sums
// of BF16 parts. k_split3 writes each operand as three BF16 planes,
// a = a1 + a2 + a3 exactly (8 + 8 + 8 significant bits, each part the
// nearest BF16 of what is left), and k_gemm_umma32 adds six of the nine
// plane products: a1 b1; a1 b2 + a2 b1; a2 b2 + a1 b3 + a3 b1. The three it
// leaves out reach 2^-24 of |a b| at worst (|a2| up to 2^-8 and |a3| up to 2^-17
// of |a|; all a in [1, 2) with b = a: 0.991 2^-24 at 0x1.00ff8p+0), FP32's own
// rounding of the product, and are mostly below a quarter of that.
//
// Accumulation. The tensor cores' FP32 accumulator cuts instead of rounding
// and a long sum in it drifts, so no sum is longer than one K block of 64
// there: the five small products first (together about 2^-7 of the leading
// one, so their twenty cuts are small), then a1 b1, in four cuts; the epilogue
// warps read the block out and add it to their registers with rounded FP32
// adds. Two accumulators alternate by block. The cuts have one sign, so sums of
// terms of one sign come out low, by about 1.2 2^-24 of their value, whatever
// K; rounded FP32 sums have no bias and grow instead. Error in 2^-24 of |X||Y|,
// root mean square (maximum), here and with the library's FP32 GEMM:
//   K       normal operands           uniform in (0, 1)
//   16      0.29 (1.9)  0.36 (2.4)    0.86 (2.0)  0.71 (3.0)
//   32      0.26 (1.9)  0.46 (4.6)    0.96 (2.9)  1.42 (7.1)
//   64      0.25 (2.0)  0.47 (3.8)    1.31 (3.8)  1.93 (8.6)
//   300     0.13 (1.0)  0.47 (4.6)    1.34 (3.7)  4.45 (20)
//   1024    0.08 (0.6)  0.15 (1.0)    1.43 (4.1)  1.16 (5.3)
//   2048    0.06 (0.4)  0.12 (0.7)    1.46 (4.6)  1.33 (5.7)
//   8192    0.04 (0.3)  0.10 (0.5)    1.52 (5.1)  1.62 (7.6)
// (from K = 512 on the library splits K at these sizes).
// Products of fewer than kSplitK terms stay with the library (gemm.cuh).
//
// Layout: 128 x BN tiles (BN 256, or 128 where that leaves SMs idle), K
// blocks of 64. One thread issues all products, so their number counts:
// 24 tcgen05.mma a block, 128 clocks each at N = 256 but 64 at N = 128, which
// is also bound by shared memory (operand reads and TMA writes, 187 bytes per
// clock against 141 at N = 256). Descriptors are a constant plus an address.
// Every plane tile of a block has its own full / empty mbarriers, and the
// products are ordered so that a plane's slot is free as early as possible:
// with N = 256, a1, b1, a2 and a3 have two slots, b2 and b3 one (224 KB); with
// N = 128 all have two (192 KB).
//
//   warp 0      lane 0 issues the TMA loads
//   warp 1      owns the TMEM; lane 0 issues the products
//   others      the epilogue, BN / 16 warps: warp w reads TMEM lanes
//               32 (w % 4) .. + 31 and 64 columns (64 sums a thread). While they
//               store a tile, the next one's first two K blocks are multiplied.
//
// A work item is a tile and one of S contiguous ranges of its K blocks. With
// S > 1 every item writes its FP32 partial tile, and the last of a tile's S
// items to finish (a ticket; no block waits for another) adds the S partials
// in range order and evaluates the remainder.
//
// Measured with sigmoid(s X Y + W) at 2048 x 1536 x 2048: 93 us (107 with
// 128-column tiles only and descriptors computed per product), against 268 us
// for the library's FP32 GEMM and the element-wise pass after it; the
// product's error against 64 bits is smaller (maximum of the result 8.7e-8
// against 1.0e-7 at K = 2048, 9.0e-8 against 1.6e-7 at K = 700).
//
// Operands with an infinity, a NaN, a magnitude of 2^60 or more or a nonzero
// one below 2^-100 (its parts would be subnormal) are not computed this way:
// k_split3 marks the tile rows or columns of the product that one lies in, and
// their tiles are computed after the others, with FP32 fma from the operands
// themselves. Below 2^60 a product is below 2^120
// and a K block's 64 of them, with the small products, below 2^127, so the
// accumulator stays finite: a1 b2 and a2 b1 have either sign, and one of them
// at -Inf beside a1 b1 at +Inf would give NaN where FP32 gives an infinity.
// What overflows later does so in the rounded FP32 adds, as in FP32. Every
// wait is bounded as in umma.cuh.
#pragma once

#include "umma.cuh"

namespace fx {
namespace umma32 {

using umma::fence_after;
using umma::fence_before;

constexpr int BM = 128, BK = 64, UK = 16;
constexpr int UNIT = 128 * BK * 2;  // shared memory of 128 rows of a plane's block
constexpr int NP = 6;               // plane tiles of a K block
constexpr int NC = 64;              // columns an epilogue thread sums
enum Plane : int { A1 = 0, A2 = 1, A3 = 2, B1 = 3, B2 = 4, B3 = 5 };

// Slots of the planes for tiles of BN columns. Plane p of K block g is in slot
// g % depth(p); its barriers are bar(p, g), its memory at at(p, g), and it is
// the use(p, g)-th block there.
template <int BN> struct Slots32 {
  static constexpr int units(int p) { return p >= B1 ? BN / 128 : 1; }
  FX_HD static constexpr uint32_t depth(int p) { return BN == 256 && (p == B2 || p == B3) ? 1 : 2; }
  FX_HD static constexpr uint32_t base(int p) {
    uint32_t u = 0;
    for (int q = 0; q < p; ++q) u += depth(q) * uint32_t(q >= B1 ? BN / 128 : 1);
    return u * uint32_t(UNIT);
  }
  FX_HD static constexpr uint32_t pick(int p, uint32_t g) { return depth(p) == 2 ? g & 1u : 0u; }
  FX_HD static constexpr uint32_t use(int p, uint32_t g) { return depth(p) == 2 ? g >> 1 : g; }
  FX_HD static constexpr uint32_t bar(int p, uint32_t g) { return uint32_t(p) * 2u + pick(p, g); }
  FX_HD static constexpr uint32_t at(int p, uint32_t g) {
    return base(p) + pick(p, g) * uint32_t(UNIT) * uint32_t(p >= B1 ? BN / 128 : 1);
  }
  static constexpr uint32_t bytes = base(NP);
  static constexpr int EPI_WARPS = BN / 16, THREADS = 64 + 32 * EPI_WARPS;
  // The order in which the producer loads a block's planes: a plane whose
  // slot frees late does not hold up one that is free.
  FX_HD static constexpr int order(int i) {
    constexpr int o256[NP] = {A3, A1, B1, A2, B3, B2}, o128[NP] = {A3, B3, A2, B2, A1, B1};
    return BN == 256 ? o256[i] : o128[i];
  }
};

struct Maps {
  CUtensorMap m[NP];  // indexed by Plane
};
// An operand as the tree binds it: element (row, k) of A and (col, k) of B at
// p[row * s_mn + k * s_k].
struct Source {
  const float* p;
  int64_t s_mn, s_k;
};
struct Bars {
  uint64_t full[2 * NP], empty[2 * NP];
  uint64_t accf[2], acce[2];  // accumulator complete / read out (one arrival per warp)
  uint64_t drain;
  uint32_t taddr;
  volatile int abort;
  int last;                   // this item completes its tile
};

// ---------------------------------------------------------------- planes

FX_D bool unsplittable(float a) {
  const uint32_t b = __float_as_uint(a) & 0x7FFFFFFFu;
  return b - 0x0D800000u >= 0x5D800000u - 0x0D800000u && b != 0u;  // not in [2^-100, 2^60), not 0
}

struct SplitArgs {
  const float* src;
  bf16* dst;          // plane p at dst + p * ldp * d1
  int64_t d0, d1;     // contiguous extent, columns
  int64_t ld, ldp;    // ldp a multiple of 8
  int64_t items;      // 8-row pieces: ceil(d0 / 8) * d1
  FastDiv per_col;    // pieces of a column
  int vec;            // every full piece is 16-byte aligned
  unsigned int* marks;  // the operand's tiles that hold an unsplittable value
  int mn_rows, shift;   // tile of element (row, column): (mn_rows ? row : column) >> shift
};

// Both operands in one launch, 8 rows of a column per thread: 32 bytes read,
// three 16-byte stores. Reads 4 and writes 6 bytes an element; bound by
// memory (the planes of the sizes this serves stay in L2 for the product).
// Rows of a piece beyond d0 (ldp's padding) are written as zeros.
static __global__ void __launch_bounds__(256) k_split3(const SplitArgs a, const SplitArgs b,
                                                       unsigned int* any) {
  const int64_t n = a.items + b.items;
  for (int64_t i = int64_t(blockIdx.x) * 256 + threadIdx.x; i < n; i += int64_t(gridDim.x) * 256) {
    const bool first = i < a.items;
    const SplitArgs& o = first ? a : b;
    const uint32_t q = uint32_t(first ? i : i - a.items);
    const uint32_t c = o.per_col.div(q);
    const int64_t r = int64_t(q - c * o.per_col.d) * 8;
    const float* s = o.src + r + int64_t(c) * o.ld;
    float x[8];
    if (o.vec && r + 8 <= o.d0) {
      Raw<float, 4> u, v;
      vload(u, s);
      vload(v, s + 4);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        x[j] = u.v[j];
        x[4 + j] = v.v[j];
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = r + j < o.d0 ? sload(s + j) : 0.0f;
    }
    Raw<bf16, 8> p1, p2, p3;
    bool bad = false;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      bad |= unsplittable(x[j]);
      p1.v[j] = __float2bfloat16_rn(x[j]);
      const float e = x[j] - __bfloat162float(p1.v[j]);
      p2.v[j] = __float2bfloat16_rn(e);
      p3.v[j] = __float2bfloat16_rn(e - __bfloat162float(p2.v[j]));
    }
    bf16* d = o.dst + r + int64_t(c) * o.ldp;
    const int64_t plane = o.ldp * o.d1;
    *reinterpret_cast<Raw<bf16, 8>*>(d) = p1;
    *reinterpret_cast<Raw<bf16, 8>*>(d + plane) = p2;
    *reinterpret_cast<Raw<bf16, 8>*>(d + 2 * plane) = p3;
    if (bad) {  // every writer stores the same value
      *any = 1u;
      o.marks[(o.mn_rows ? r : int64_t(c)) >> o.shift] = 1u;
    }
  }
}

// ---------------------------------------------------------------- product

template <int BN, bool AMN, bool BMN> FX_HD constexpr uint32_t idesc() {  // BF16 in, FP32 out
  return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(AMN) << 15) | (uint32_t(BMN) << 16) |
         (uint32_t(BN >> 3) << 17) | (uint32_t(BM >> 4) << 24);
}

// One plane tile: rows mn0 .. mn0 + ROWS - 1 of the operand, K block k0.
template <bool MNMAJOR, int ROWS>
FX_D void load_plane(char* dst, const CUtensorMap* m, int mn0, int k0, uint64_t* bar) {
  tma::arrive_expect_tx(bar, uint32_t(ROWS * BK * 2));
  if (MNMAJOR) {
#pragma unroll
    for (int j = 0; j < ROWS / 64; ++j) tma::load_2d(dst + j * (UNIT / 2), m, mn0 + 64 * j, k0, bar);
  } else {
    tma::load_2d(dst, m, k0, mn0, bar);
  }
}
// The matrix descriptor of a plane tile at shared address 0, and its step per
// 16 of K, in the descriptor's 16-byte units.
template <bool MNMAJOR> FX_D uint64_t plane_desc() {
  return umma::desc(0, MNMAJOR ? UNIT / 2 : 16, 1024);
}
template <bool MNMAJOR> FX_HD constexpr uint32_t kstep() { return (MNMAJOR ? UK * 128 : UK * 2) / 16; }

// A thread's row m of Z, columns n0 .. n0 + NC - 1, from the product values acc;
// the other leaves' values are loaded one piece of 8 columns ahead.
template <class T, class E, int PS>
FX_D void store_row(const E& e, const Slots& sl, float* z, int64_t ldz, int64_t m, int n0, int N,
                    const float (&acc)[NC]) {
  using LL = leaves_t<E>;
  constexpr int NL = tl_size<LL>::value, CW = 8;
  T wn[NL][CW], wc[NL][CW];
  if (n0 < N) umma::load_others<LL, PS, T, CW>(wn, sl, m, n0, N - n0 < CW ? N - n0 : CW);
#pragma unroll
  for (int c = 0; c < NC / CW; ++c) {
    const int nc = n0 + c * CW;
    if (nc < N) {
      const int nn = N - nc < CW ? N - nc : CW;
#pragma unroll
      for (int l = 0; l < NL; ++l)
#pragma unroll
        for (int j = 0; j < CW; ++j) wc[l][j] = wn[l][j];
      const int nx = nc + CW;
      if (c + 1 < NC / CW && nx < N)
        umma::load_others<LL, PS, T, CW>(wn, sl, m, nx, N - nx < CW ? N - nx : CW);
#pragma unroll
      for (int j = 0; j < CW; ++j) {
        if (j < nn) {
          umma::ECtx<LL, PS, T, CW> cx{wc, acc[c * CW + j], j};
          sstore(z + m + int64_t(nc + j) * ldz, e.ev(cx));
        }
      }
    }
  }
}

// Brings the other leaves' part of a tile towards L2 while it is multiplied:
// thread i of the epilogue takes half a column (256 bytes).
template <class LL, int PS, int I = 0>
FX_D void prefetch_others(const Slots& sl, int64_t m, int64_t n, int M) {
  if constexpr (I < tl_size<LL>::value) {
    using L = typename tl_at<LL, I>::type;
    if constexpr (L::slot != PS) {
      const SlotView& s = sl.s[L::slot];
      const float* p = static_cast<const float*>(s.p) + m + n * s.ld;
#pragma unroll
      for (int j = 0; j < 64; j += 32)
        if (m + j < M) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + j));
    }
    prefetch_others<LL, PS, I + 1>(sl, m, n, M);
  }
}

// Barrier 1 over the block's NT epilogue threads; true if v is for all of them.
template <int NT> FX_D bool all_of(bool v) {
  uint32_t r;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.and.pred q, 1, %2, p;\n"
      "selp.u32 %0, 1, 0, q;\n}"
      : "=r"(r)
      : "r"(uint32_t(v)), "n"(NT)
      : "memory");
  return r != 0;
}

// Tiles with unsplittable values: any[0] is set when there are some, then
// rows[tile row] and cols[tile column] hold the marks; any[1] counts blocks.
struct Marks {
  unsigned int *any, *rows, *cols;
  FX_D bool direct(int tm, int tn) const { return (rows[tm] | cols[tn]) != 0u; }
};

// The product of the marked tiles by FP32 fma from the operands themselves:
// 64 x 128 pieces, each by NG groups of 256 threads that take every NG-th K step
// of 16 and add their sums at the end; 4 x 8 results a thread, two K steps on
// their way by cp.async while one is multiplied from shared memory. Bound by
// instruction issue, half of it fma, and with few marked tiles by the SMs that
// have a piece. Microseconds with one element out of range, and with one in every
// tile row (in brackets the loop before, which took all tiles for one element: 8
// x 8 results by 256 threads that waited for each step's loads; then the
// library's FP32 GEMM and the element-wise pass after it):
//   2048 x 1536 x 2048  229, 490 (1432; 262)    1000^3          125, 103 (248; 43)
//   3000^3              495, 1790 (4338; 840)   512 x 512 x 4096  368, 338 (974; 54)
// (The next step held in registers instead spilled: 557 for 490; fma.rn.f32x2 was
// no faster, 8 x 8 results by 256 threads slower.)
template <int BN> struct Fma32 {
  static_assert(BN == 128 || BN == 256, "one or two groups (barriers 2 and 3)");
  static constexpr int NG = BN / 128, NT = 256 * NG;  // the block has more threads: the rest leave
  static constexpr int RM = 4, RN = 8, TM = 16 * RM, TN = 16 * RN, KS = 16;
  static constexpr int LA = TM + 4, LB = TN + 4;      // shared-memory rows of one k
  static constexpr int ST = 3, STAGE = KS * (LA + LB), GROUP = ST * STAGE;
  static constexpr int PIECES = (BM / TM) * (BN / TN);  // of a tile
  static_assert(NG * GROUP * 4 <= int(Slots32<BN>::bytes) && (NG - 1) * TM * TN * 4 <= int(Slots32<BN>::bytes),
                "shared memory");
};
// A thread's elements of a ROWS x 16 step of an operand: i = t, t + 256, ...,
// counted along the operand's contiguous dimension.
template <int ROWS, int LD, int STEP> struct FmaWalk {
  static constexpr int KS = 16, N = ROWS * KS / 256;
  const float* p;      // the first one of the next step
  int64_t dp, dk;      // to the next one, to the next step
  int at, da, k, kj;   // place in the staged step, its step; k of the first one and its step
  uint32_t inside;     // bit j: row of element j is inside the operand
  FX_D FmaWalk(const Source& s, int r0, int R, int k0, int t) {
    const bool mn = s.s_mn == 1;
    const int r = mn ? t % ROWS : t / KS, dr = mn ? 0 : 256 / KS;
    k = mn ? t / ROWS : t % KS;
    kj = mn ? 256 / ROWS : 0;
    p = s.p + (r0 + r) * s.s_mn + (k0 + k) * s.s_k;
    dp = dr * s.s_mn + kj * s.s_k;
    dk = int64_t(STEP) * s.s_k;
    at = k * LD + r;
    da = kj * LD + dr;
    inside = 0u;
#pragma unroll
    for (int j = 0; j < N; ++j) inside |= uint32_t(r0 + r + j * dr < R) << j;
  }
  FX_D void copy(float* step, int k0, int K) {  // zeros beyond R and K
    const uint32_t q = tma::saddr(step + at);
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const bool in = (inside >> j & 1u) && (k0 + KS <= K || k0 + k + j * kj < K);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(q + 4u * uint32_t(j * da)),
                   "l"(p + j * dp), "r"(in ? 4u : 0u)
                   : "memory");
    }
    p += dk;
  }
};

// Columns n0 .. n0 + TN - 1 of rows m0 .. m0 + TM - 1 of Z.
template <int BN, class E, int PS>
FX_D void fma_piece(char* smem, const E& e, const Slots& sl, float* z, int64_t ldz, int M, int N,
                    int K, const Source& A, const Source& B, int m0, int n0) {
  using LL = leaves_t<E>;
  using F = Fma32<BN>;
  constexpr int NL = tl_size<LL>::value, KS = F::KS, RM = F::RM, RN = F::RN;
  const int grp = threadIdx.x / 256, t = threadIdx.x % 256;
  const int tx = t % 16, ty = t / 16;  // rows 4 tx .. + 3, columns 4 ty .. + 3 and 64 + 4 ty .. + 3
  float* base = reinterpret_cast<float*>(smem) + grp * F::GROUP;
  float* sums = reinterpret_cast<float*>(smem);
  auto group_sync = [&]() {
    if (grp == 0) asm volatile("bar.sync 2, 256;" ::: "memory");
    else asm volatile("bar.sync 3, 256;" ::: "memory");
  };
  auto all_sync = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(F::NT) : "memory"); };
  float acc[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) acc[i][j] = 0.0f;
  const int k0 = grp * KS, steps = K > k0 ? (K - k0 + KS * F::NG - 1) / (KS * F::NG) : 0;
  FmaWalk<F::TM, F::LA, KS * F::NG> wa(A, m0, M, k0, t);
  FmaWalk<F::TN, F::LB, KS * F::NG> wb(B, n0, N, k0, t);
  auto fetch = [&](int i) {  // step i, into slot i % ST
    if (i < steps) {
      float* step = base + i % F::ST * F::STAGE;
      wa.copy(step, k0 + i * KS * F::NG, K);
      wb.copy(step + KS * F::LA, k0 + i * KS * F::NG, K);
    }
    cpa::commit();
  };
#pragma unroll
  for (int i = 0; i < F::ST - 1; ++i) fetch(i);
  for (int i = 0; i < steps; ++i) {
    cpa::wait_pending<F::ST - 2>();
    group_sync();  // step i has landed for all, and all have read the slot that is filled next
    fetch(i + F::ST - 1);
    const float* sa = base + i % F::ST * F::STAGE;
    const float* sb = sa + KS * F::LA;
#pragma unroll 2
    for (int k = 0; k < KS; ++k) {  // beyond K both operands are zeros
      const float4 a0 = *reinterpret_cast<const float4*>(sa + k * F::LA + 4 * tx);
      const float4 b0 = *reinterpret_cast<const float4*>(sb + k * F::LB + 4 * ty);
      const float4 b1 = *reinterpret_cast<const float4*>(sb + k * F::LB + 64 + 4 * ty);
      const float a[RM] = {a0.x, a0.y, a0.z, a0.w}, b[RN] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) acc[i][j] = __fmaf_rn(a[i], b[j], acc[i][j]);
    }
  }
  cpa::wait_pending<0>();
  if (F::NG > 1) {  // group 0 adds the other group's sums
    all_sync();     // the staged steps are read
    if (grp > 0) {
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) sums[(i * RN + j) * 256 + t] = acc[i][j];
    }
    all_sync();
    if (grp == 0) {
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) acc[i][j] += sums[(i * RN + j) * 256 + t];
    }
  }
  if (grp == 0) {
#pragma unroll
    for (int j = 0; j < RN; ++j) {
      const int n = n0 + (j / 4) * 64 + 4 * ty + j % 4;
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        const int m = m0 + 4 * tx + i;
        if (m < M && n < N) {
          float w[NL][1];
          umma::load_others<LL, PS, float, 1>(w, sl, m, n, 1);
          umma::ECtx<LL, PS, float, 1> cx{w, acc[i][j], 0};
          sstore(z + m + int64_t(n) * ldz, e.ev(cx));
        }
      }
    }
  }
  all_sync();  // the next piece's first step overwrites the sums
}

// Every marked tile's pieces, dealt out to the blocks in order. Each warp finds
// the marked tiles for itself, 32 at a time.
template <int BN, class E, int PS>
FX_D void fma_tiles(char* smem, const E& e, const Slots& sl, float* z, int64_t ldz, int M, int N,
                    int K, const Source& A, const Source& B, const Marks& marks, int tiles_m, int tiles_n) {
  using F = Fma32<BN>;
  if (threadIdx.x >= F::NT) return;
  const int ntiles = tiles_m * tiles_n, lane = threadIdx.x % 32;
  int64_t next = blockIdx.x, seen = 0;  // this block's next piece, pieces of the tiles so far
  for (int base = 0; base < ntiles; base += 32) {
    const int t = base + lane;
    uint32_t found = __ballot_sync(0xffffffffu, t < ntiles && marks.direct(t % tiles_m, t / tiles_m));
    for (; found != 0u; found &= found - 1u, seen += F::PIECES) {
      const int tile = base + __ffs(int(found)) - 1;
      for (; next < seen + F::PIECES; next += gridDim.x) {
        const int q = int(next - seen), m0 = tile % tiles_m * BM + q % (BM / F::TM) * F::TM;
        const int n0 = tile / tiles_m * BN + q / (BM / F::TM) * F::TN;
        if (m0 < M && n0 < N) fma_piece<BN, E, PS>(smem, e, sl, z, ldz, M, N, K, A, B, m0, n0);
      }
    }
  }
}

template <int BN, bool AMN, bool BMN, class E, int PS>
__global__ void __launch_bounds__(Slots32<BN>::THREADS, 1)
    k_gemm_umma32(const __grid_constant__ Maps maps, const E e, const Slots sl, float* z,
                  const int64_t ldz, const int M, const int N, const int K, const int S,
                  float* part, unsigned int* tickets, const Marks marks, const Source srcA,
                  const Source srcB, unsigned int* err) {
  using SL = Slots32<BN>;
  extern __shared__ char smem_raw[];
  char* smem = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                       ~uintptr_t(1023));
  Bars& bars = *reinterpret_cast<Bars*>(smem + SL::bytes);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int tiles_m = (M + BM - 1) / BM, tiles_n = (N + BN - 1) / BN;
  const int ntiles = tiles_m * tiles_n;
  const int nitems = ntiles * S;
  const int nk = (K + BK - 1) / BK;
  const bool any = __ldcg(marks.any) != 0u;  // the same for every thread of the grid
  auto direct = [&](int tm, int tn) { return any && marks.direct(tm, tn); };
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2 * NP; ++i) {
      tma::mbar_init(&bars.full[i], 1);
      tma::mbar_init(&bars.empty[i], 1);
    }
    for (int b = 0; b < 2; ++b) {
      tma::mbar_init(&bars.accf[b], 1);
      tma::mbar_init(&bars.acce[b], SL::EPI_WARPS);
    }
    tma::mbar_init(&bars.drain, 1);
    bars.abort = 0;
    tma::fence_mbar_init();
  }
  if (warp == 1) {
    umma::tmem_alloc(&bars.taddr, 2 * BN);
    umma::tmem_relinquish();
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tbase = bars.taddr;

  if (warp == 0) {
    if (lane == 0) {
      uint32_t g = 0;   // K blocks so far
      uint32_t gf = 0;  // where the producer gave up: block and position in the order
      int pf = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
        const int s = it / ntiles;
        int tm, tn;
        umma::tile_of(it - s * ntiles, tiles_m, tiles_n, tm, tn);
        if (direct(tm, tn)) continue;
        const int m0 = tm * BM, n0 = tn * BN;
        const int kb1 = int(int64_t(nk) * (s + 1) / S);
        for (int kb = int(int64_t(nk) * s / S); kb < kb1 && ok; ++kb, ++g) {
          const int k0 = kb * BK;
#pragma unroll
          for (int o = 0; o < NP; ++o) {
            const int p = SL::order(o);
            const uint32_t i = SL::bar(p, g), use = SL::use(p, g);
            if (ok && use >= 1 && !tma::wait(&bars.empty[i], (use - 1u) & 1u, err)) {
              ok = false;
              gf = g;
              pf = o;
            }
            if (!ok) continue;
            if (p >= B1) load_plane<BMN, BN>(smem + SL::at(p, g), &maps.m[p], n0, k0, &bars.full[i]);
            else load_plane<AMN, BM>(smem + SL::at(p, g), &maps.m[p], m0, k0, &bars.full[i]);
          }
        }
      }
      if (!ok) {  // wait (bounded) for the copies still in flight
        bars.abort = 1;
        for (int o = 0; o < NP; ++o) {
          const int p = SL::order(o);
          const uint32_t n = gf + (o < pf ? 1u : 0u);  // blocks whose plane p was issued
          for (uint32_t j = n > SL::depth(p) ? n - SL::depth(p) : 0u; j < n; ++j)
            tma::wait(&bars.full[SL::bar(p, j)], SL::use(p, j) & 1u, nullptr);
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t ID = idesc<BN, AMN, BMN>();
      const uint64_t da = plane_desc<AMN>(), db = plane_desc<BMN>();
      const uint32_t s16 = tma::saddr(smem) >> 4;
      uint32_t g = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
        const int s = it / ntiles;
        const int nkb = int(int64_t(nk) * (s + 1) / S) - int(int64_t(nk) * s / S);
        if (any) {
          int tm, tn;
          umma::tile_of(it - s * ntiles, tiles_m, tiles_n, tm, tn);
          if (direct(tm, tn)) continue;
        }
        for (int kb = 0; kb < nkb && ok; ++kb, ++g) {
          const uint32_t acc = tbase + (g & 1u) * BN;
          auto ready = [&](int p) {
            if (ok && !tma::wait(&bars.full[SL::bar(p, g)], SL::use(p, g) & 1u, err)) ok = false;
          };
          auto release = [&](int p) { umma::commit(&bars.empty[SL::bar(p, g)]); };
          auto product = [&](int pa, int pb, bool fresh) {
            const uint64_t a = da | uint64_t(s16 + (SL::at(pa, g) >> 4));
            const uint64_t b = db | uint64_t(s16 + (SL::at(pb, g) >> 4));
#pragma unroll
            for (int k = 0; k < BK / UK; ++k)
              umma::mma(acc, a + uint32_t(k) * kstep<AMN>(), b + uint32_t(k) * kstep<BMN>(), ID,
                        (!fresh || k > 0) ? 1u : 0u);
          };
          // the epilogue has read out the block this accumulator held before
          if (g >= 2 && !tma::wait(&bars.acce[g & 1u], ((g >> 1) - 1u) & 1u, err)) ok = false;
          ready(A3);
          ready(B1);
          if (!ok) break;
          fence_after();
          product(A3, B1, true);
          release(A3);
          ready(A1);
          ready(B3);
          if (!ok) break;
          fence_after();
          product(A1, B3, false);
          release(B3);
          ready(A2);
          if (!ok) break;
          fence_after();
          product(A2, B1, false);
          ready(B2);
          if (!ok) break;
          fence_after();
          product(A1, B2, false);
          product(A2, B2, false);
          release(A2);
          release(B2);
          product(A1, B1, false);
          release(A1);
          release(B1);
          umma::commit(&bars.accf[g & 1u]);
        }
      }
      if (!ok) {  // wake the epilogue (it sees the abort) after what was issued
        bars.abort = 1;
        umma::commit(&bars.accf[0]);
        umma::commit(&bars.accf[1]);
      }
      umma::commit(&bars.drain);
      tma::wait(&bars.drain, 0u, err);
    }
    __syncwarp();
  } else {
    const int q = warp & 3;                // TMEM lane quarter
    const int col = (warp - 2) / 4 * NC;   // first of the thread's columns
    const uint32_t tmine = tbase + (uint32_t(q * 32) << 16) + uint32_t(col);
    const int row = q * 32 + lane;
    uint32_t g = 0;
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
      const int s = it / ntiles, t = it - s * ntiles;
      const int nkb = int(int64_t(nk) * (s + 1) / S) - int(int64_t(nk) * s / S);
      bool ready = true;
      int tm, tn;
      umma::tile_of(t, tiles_m, tiles_n, tm, tn);
      if (direct(tm, tn)) continue;
      if (s == S - 1) {
        const int i = int(threadIdx.x) - 64, n = tn * BN + i / 2;
        if (n < N) prefetch_others<leaves_t<E>, PS>(sl, int64_t(tm) * BM + (i & 1) * 64, n, M);
      }
      float acc[NC];
#pragma unroll
      for (int j = 0; j < NC; ++j) acc[j] = 0.0f;
      for (int kb = 0; kb < nkb; ++kb, ++g) {
        const uint32_t b = g & 1u;
        ready = tma::wait(&bars.accf[b], (g >> 1) & 1u, err);
        fence_after();
        // the TMEM loads are warp-wide: the warp decides together
        ready = __all_sync(0xffffffffu, ready && !bars.abort);
        if (!ready) break;
#pragma unroll
        for (int c = 0; c < NC / 16; ++c) {
          uint32_t r[16];
          umma::ld16(tmine + b * BN + uint32_t(c * 16), r);
          umma::wait_ld();
#pragma unroll
          for (int j = 0; j < 16; ++j) acc[c * 16 + j] += __uint_as_float(r[j]);
        }
        fence_before();
        __syncwarp();
        if (lane == 0) tma::arrive(&bars.acce[b]);
      }
      if (S == 1 && !ready) break;
      if (S > 1) {
        float* mine = part + int64_t(it) * (BM * BN) + col * BM + row;
        if (ready) {
#pragma unroll
          for (int j = 0; j < NC; ++j) __stcg(mine + j * BM, acc[j]);
        }
        __threadfence();
        // a warp that gave up its wait still comes here: the warps leave
        // together, and none is left at a barrier that another never reaches
        if (!all_of<32 * SL::EPI_WARPS>(ready)) break;
        if (warp == 2 && lane == 0) bars.last = atomicAdd(tickets + t, 1u) == unsigned(S - 1);
        asm volatile("bar.sync 1, %0;" ::"n"(32 * SL::EPI_WARPS) : "memory");
        if (!bars.last) continue;
        __threadfence();
        if (warp == 2 && lane == 0) tickets[t] = 0u;  // ready for the next launch
#pragma unroll
        for (int j = 0; j < NC; ++j) acc[j] = 0.0f;
        for (int k = 0; k < S; ++k) {
          const float* p = part + (int64_t(k) * ntiles + t) * (BM * BN) + col * BM + row;
#pragma unroll
          for (int j = 0; j < NC; ++j) acc[j] += __ldcg(p + j * BM);
        }
      }
      const int64_t m = int64_t(tm) * BM + row;
      if (m < M) store_row<float, E, PS>(e, sl, z, ldz, m, tn * BN + col, N, acc);
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    umma::tmem_dealloc(tbase, 2 * BN);
  }
  if (!any) return;
  // no copy and no product is in flight: the shared memory is free, unless a
  // wait was given up (recorded; the result is void)
  if (!bars.abort)
    fma_tiles<BN, E, PS>(smem, e, sl, z, ldz, M, N, K, srcA, srcB, marks, tiles_m, tiles_n);
  // the last block clears the marks for the next launch
  __syncthreads();
  if (threadIdx.x == 0) bars.last = atomicAdd(marks.any + 1, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!bars.last) return;
  for (int i = threadIdx.x; i < tiles_m + tiles_n; i += blockDim.x)
    (i < tiles_m ? marks.rows[i] : marks.cols[i - tiles_m]) = 0u;
  if (threadIdx.x == 0) marks.any[0] = marks.any[1] = 0u;
}

// Tile width and K ranges per tile: the pair that minimises waves of work
// items times their length, in K blocks of a 128-column tile. An item costs
// its own blocks (two units each at 256 columns) and about two to fill and
// drain its pipeline, and with S > 1 one more to write its partial tile, per
// 128 columns, and S to add them up.
struct Shape32 {
  int bn, S;
};
inline Shape32 choose_shape(int64_t M, int64_t N, int nk, int sms) {
  Shape32 best{256, 1};
  int64_t cost = -1;
  for (int bn : {256, 128}) {
    const int64_t ntiles = ((M + BM - 1) / BM) * ((N + bn - 1) / bn);
    for (int S = 1; S <= 16 && S <= nk; ++S) {
      const int64_t waves = (ntiles * S + sms - 1) / sms, w = bn / 128;
      // products at 128 columns run at about 3/4 of the rate
      const int64_t blocks = int64_t((nk + S - 1) / S) * (bn == 256 ? 6 : 4);
      const int64_t c = waves * (blocks + 8) + (S > 1 ? (waves + S) * 2 * w : 0);
      if (cost < 0 || c < cost) {
        cost = c;
        best = Shape32{bn, S};
      }
    }
  }
  return best;
}

}  // namespace umma32
}  // namespace fx
