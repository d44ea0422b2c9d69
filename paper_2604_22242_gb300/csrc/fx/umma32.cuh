// umma32.cuh - an FP32 matrix product on the fifth-generation tensor cores,
// with the tree's element-wise remainder evaluated in its epilogue.
//
// The tensor cores multiply 16-bit operands; FP32 operands run there as sums
// of BF16 parts. k_split3 writes each operand as three BF16 planes,
// a = a1 + a2 + a3 exactly (8 + 8 + 8 significant bits, each part the
// nearest BF16 of what is left), and k_gemm_umma32 adds six of the nine
// plane products: a1 b1; a1 b2 + a2 b1; a2 b2 + a1 b3 + a3 b1. The three it
// leaves out are below 2^-26 of |a b|, a quarter of FP32's own rounding of
// the product.
//
// Accumulation. The tensor cores' FP32 accumulator cuts instead of rounding
// and a long sum in it drifts, so no sum of leading products (a1 b1) is
// longer than one K block of 64 there: the epilogue warps read it out and
// add it to their registers with rounded FP32 adds. The five small products,
// at most 2^-8 of the leading one, keep one accumulator for the whole tile.
//
// Layout: 128 x 128 tiles, K blocks of 64. A block is six 16 KB plane tiles
// (a3 b1 a1 b3 a2 b2, in the order of their first use); two blocks are in
// shared memory, every plane tile with its own full / empty mbarriers, so a
// plane's slot refills as soon as its last product has read it. Per SM and
// block: 96 KB from L2 for 24 tcgen05.mma of 128 x 128 x 16, 64 bytes per
// clock at the tensor cores' rate (a BF16 product with 128 x 256 tiles needs
// 96). TMEM (512 columns): two leading accumulators, alternating by K block,
// and two small-product accumulators, alternating by tile.
//
//   warp 0      lane 0 issues the TMA loads
//   warp 1      owns the TMEM; lane 0 issues the products
//   warps 2-9   the epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31, the
//               first four warps columns 0-63 of the tile, the others 64-127
//               (64 sums a thread; 128 would spill at ten warps). While they
//               store a tile, the next one's first two K blocks are multiplied.
//
// A work item is a tile and one of S contiguous ranges of its K blocks. With
// S > 1 every item writes its FP32 partial tile, and the last of a tile's S
// items to finish (a ticket; no block waits for another) adds the S partials
// in range order and evaluates the remainder.
//
// Measured with sigmoid(s X Y + W) at 2048 x 1536 x 2048: 107 us, against
// 268 us for the library's FP32 GEMM and the element-wise pass after it; the
// product's error against 64 bits is smaller (maximum of the result 8.7e-8
// against 1.0e-7 at K = 2048, 9.0e-8 against 1.6e-7 at K = 700).
//
// Operands with an infinity, a NaN, a magnitude of 2^127 or more (it could
// round up to a BF16 infinity) or a nonzero one below 2^-100 (its parts would
// be subnormal) cannot be split this way: k_split3 records one in a flag and
// every block then computes its tiles with FP32 fma from the operands
// themselves. Every wait is bounded as in umma.cuh.
#pragma once

#include "umma.cuh"

namespace fx {
namespace umma32 {

using umma::fence_after;
using umma::fence_before;

constexpr int BM = 128, BN = 128, BK = 64, UK = 16;
constexpr int TILE = BM * BK * 2;  // one plane tile of either operand
constexpr int NP = 6;              // plane tiles of a K block
constexpr int EPI_WARPS = 8;
constexpr int NC = BN / 2;         // columns an epilogue thread sums
constexpr int THREADS = 64 + 32 * EPI_WARPS;
enum Plane : int { A3 = 0, B1 = 1, A1 = 2, B3 = 3, A2 = 4, B2 = 5 };

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
  uint64_t full[2][NP], empty[2][NP];
  uint64_t hif[2], hie[2];  // leading accumulator complete / read out (one arrival per warp)
  uint64_t loe[2];          // small-product accumulator read out (one arrival per warp)
  uint64_t drain;
  uint32_t taddr;
  volatile int abort;
  int last;                 // this item completes its tile
};

// ---------------------------------------------------------------- planes

FX_D bool unsplittable(float a) {
  const uint32_t b = __float_as_uint(a) & 0x7FFFFFFFu;
  return b - 0x0D800000u >= 0x7F000000u - 0x0D800000u && b != 0u;  // not in [2^-100, 2^127), not 0
}

struct SplitArgs {
  const float* src;
  bf16* dst;          // plane p at dst + p * ldp * d1
  int64_t d0, d1;     // contiguous extent, columns
  int64_t ld, ldp;    // ldp a multiple of 8
  int64_t items;      // 8-row pieces: ceil(d0 / 8) * d1
  FastDiv per_col;    // pieces of a column
  int vec;            // every full piece is 16-byte aligned
};

// Both operands in one launch, 8 rows of a column per thread: 32 bytes read,
// three 16-byte stores. Reads 4 and writes 6 bytes an element; bound by
// memory (the planes of the sizes this serves stay in L2 for the product).
// Rows of a piece beyond d0 (ldp's padding) are written as zeros.
static __global__ void __launch_bounds__(256) k_split3(const SplitArgs a, const SplitArgs b,
                                                       unsigned int* flag) {
  bool bad = false;
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
  }
  if (bad) *flag = 1u;  // every writer stores the same value
}

// ---------------------------------------------------------------- product

FX_D void ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}

template <bool AMN, bool BMN> FX_HD constexpr uint32_t idesc() {  // kind::f16, BF16 in, FP32 out
  return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(AMN) << 15) | (uint32_t(BMN) << 16) |
         (uint32_t(BN >> 3) << 17) | (uint32_t(BM >> 4) << 24);
}

// One plane tile: rows mn0 .. mn0 + 127 of the operand, K block k0.
template <bool MNMAJOR>
FX_D void load_plane(char* dst, const CUtensorMap* m, int mn0, int k0, uint64_t* bar) {
  tma::arrive_expect_tx(bar, TILE);
  if (MNMAJOR) {
    tma::load_2d(dst, m, mn0, k0, bar);
    tma::load_2d(dst + TILE / 2, m, mn0 + 64, k0, bar);
  } else {
    tma::load_2d(dst, m, k0, mn0, bar);
  }
}
template <bool MNMAJOR> FX_D uint64_t plane_desc(uint32_t s, int k) {
  return MNMAJOR ? umma::desc(s + uint32_t(k) * UK * 128, TILE / 2, 1024)
                 : umma::desc(s + uint32_t(k) * UK * 2, 16, 1024);
}

// A thread's row m of Z, columns n0 .. n0 + NC - 1, from the product values acc;
// the other leaves' values are loaded one piece of 16 columns ahead.
template <class T, class E, int PS>
FX_D void store_row(const E& e, const Slots& sl, float* z, int64_t ldz, int64_t m, int n0, int N,
                    const float (&acc)[NC]) {
  using LL = leaves_t<E>;
  constexpr int NL = tl_size<LL>::value, CW = 16;
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

// The product by FP32 fma from the operands themselves (unsplittable values):
// 256 threads, 8 x 8 results each, K steps of 16 through shared memory.
template <class E, int PS>
FX_D void fma_tiles(char* smem, const E& e, const Slots& sl, float* z, int64_t ldz, int M, int N,
                    int K, const Source& A, const Source& B, int tiles_m, int tiles_n) {
  using LL = leaves_t<E>;
  constexpr int KS = 16, LDS = BM + 4, NL = tl_size<LL>::value;
  float* sa = reinterpret_cast<float*>(smem);
  float* sb = sa + KS * LDS;
  const int tid = threadIdx.x, tx = tid % 16, ty = (tid / 16) % 16;
  for (int t = blockIdx.x; t < tiles_m * tiles_n; t += gridDim.x) {
    int tm, tn;
    umma::tile_of(t, tiles_m, tiles_n, tm, tn);
    const int m0 = tm * BM, n0 = tn * BN;
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = 0.0f;
    for (int k0 = 0; k0 < K; k0 += KS) {
      __syncthreads();
      if (tid < 256) {
        for (int i = tid; i < KS * BM; i += 256) {
          // walk the operand along its contiguous dimension
          const int ka = A.s_mn == 1 ? i / BM : i % KS, ra = A.s_mn == 1 ? i % BM : i / KS;
          const int kb = B.s_mn == 1 ? i / BM : i % KS, rb = B.s_mn == 1 ? i % BM : i / KS;
          sa[ka * LDS + ra] = (m0 + ra < M && k0 + ka < K)
                                  ? sload(A.p + (m0 + ra) * A.s_mn + (k0 + ka) * A.s_k) : 0.0f;
          sb[kb * LDS + rb] = (n0 + rb < N && k0 + kb < K)
                                  ? sload(B.p + (n0 + rb) * B.s_mn + (k0 + kb) * B.s_k) : 0.0f;
        }
      }
      __syncthreads();
      if (tid < 256) {
        const int kn = K - k0 < KS ? K - k0 : KS;
        for (int k = 0; k < kn; ++k) {
          float a[8], b[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) a[i] = sa[k * LDS + tx + 16 * i];
#pragma unroll
          for (int j = 0; j < 8; ++j) b[j] = sb[k * LDS + ty + 16 * j];
#pragma unroll
          for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = __fmaf_rn(a[i], b[j], acc[i][j]);
        }
      }
    }
    if (tid < 256) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int m = m0 + tx + 16 * i;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int n = n0 + ty + 16 * j;
          if (m < M && n < N) {
            float w[NL][1];
            umma::load_others<LL, PS, float, 1>(w, sl, m, n, 1);
            umma::ECtx<LL, PS, float, 1> cx{w, acc[i][j], 0};
            sstore(z + m + int64_t(n) * ldz, e.ev(cx));
          }
        }
      }
    }
  }
}

template <bool AMN, bool BMN, class E, int PS>
__global__ void __launch_bounds__(THREADS, 1)
    k_gemm_umma32(const __grid_constant__ Maps maps, const E e, const Slots sl, float* z,
                  const int64_t ldz, const int M, const int N, const int K, const int S,
                  float* part, unsigned int* tickets, unsigned int* flag, const Source srcA,
                  const Source srcB, unsigned int* err) {
  extern __shared__ char smem_raw[];
  char* smem = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                       ~uintptr_t(1023));
  Bars& bars = *reinterpret_cast<Bars*>(smem + 2 * NP * TILE);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int tiles_m = (M + BM - 1) / BM, tiles_n = (N + BN - 1) / BN;
  const int ntiles = tiles_m * tiles_n;
  const int nitems = ntiles * S;
  const int nk = (K + BK - 1) / BK;
  const bool direct = __ldcg(flag) != 0u;  // the same for every thread of the grid
  __syncthreads();
  // the last block to have read the flag clears it (and its count) for the next launch
  if (threadIdx.x == 0 && atomicAdd(flag + 1, 1u) == gridDim.x - 1) {
    flag[0] = 0u;
    flag[1] = 0u;
  }
  if (direct) {
    fma_tiles<E, PS>(smem, e, sl, z, ldz, M, N, K, srcA, srcB, tiles_m, tiles_n);
    return;
  }
  if (threadIdx.x == 0) {
    for (int b = 0; b < 2; ++b) {
      for (int p = 0; p < NP; ++p) {
        tma::mbar_init(&bars.full[b][p], 1);
        tma::mbar_init(&bars.empty[b][p], 1);
      }
      tma::mbar_init(&bars.hif[b], 1);
      tma::mbar_init(&bars.hie[b], EPI_WARPS);
      tma::mbar_init(&bars.loe[b], EPI_WARPS);
    }
    tma::mbar_init(&bars.drain, 1);
    bars.abort = 0;
    tma::fence_mbar_init();
  }
  if (warp == 1) {
    umma::tmem_alloc(&bars.taddr, 512);
    umma::tmem_relinquish();
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tbase = bars.taddr;
  // leading accumulators at columns 0 and 128, small-product ones at 256 and 384

  if (warp == 0) {
    if (lane == 0) {
      uint32_t g = 0;  // K blocks so far
      bool ok = true;
      for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
        const int s = it / ntiles;
        int tm, tn;
        umma::tile_of(it - s * ntiles, tiles_m, tiles_n, tm, tn);
        const int m0 = tm * BM, n0 = tn * BN;
        const int kb1 = int(int64_t(nk) * (s + 1) / S);
        for (int kb = int(int64_t(nk) * s / S); kb < kb1 && ok; ++kb, ++g) {
          const int b = int(g & 1u);
          char* st = smem + b * NP * TILE;
          const int k0 = kb * BK;
          int p = 0;
          for (; p < NP; ++p) {
            if (g >= 2 && !tma::wait(&bars.empty[b][p], ((g >> 1) - 1u) & 1u, err)) {
              ok = false;
              break;
            }
            if (p == B1 || p == B2 || p == B3)
              load_plane<BMN>(st + p * TILE, &maps.m[p], n0, k0, &bars.full[b][p]);
            else
              load_plane<AMN>(st + p * TILE, &maps.m[p], m0, k0, &bars.full[b][p]);
          }
          if (!ok) {  // wait (bounded) for what is still in flight (here g >= 2)
            bars.abort = 1;
            for (int j = 0; j < NP; ++j) {
              tma::wait(&bars.full[b ^ 1][j], ((g - 1u) >> 1) & 1u, nullptr);
              tma::wait(&bars.full[b][j], ((g >> 1) - (j < p ? 0u : 1u)) & 1u, nullptr);
            }
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t ID = idesc<AMN, BMN>();
      uint32_t g = 0;
      int i = 0;  // items so far
      bool ok = true;
      for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x, ++i) {
        const int s = it / ntiles;
        const int kb0 = int(int64_t(nk) * s / S), kb1 = int(int64_t(nk) * (s + 1) / S);
        if (i >= 2 && !tma::wait(&bars.loe[i & 1], uint32_t((i - 2) >> 1) & 1u, err)) {
          ok = false;
          break;
        }
        const uint32_t lo = tbase + 256u + uint32_t(i & 1) * BN;
        for (int kb = kb0; kb < kb1 && ok; ++kb, ++g) {
          const int b = int(g & 1u);
          const uint32_t par = (g >> 1) & 1u;
          const uint32_t st = tma::saddr(smem + b * NP * TILE);
          const uint32_t hi = tbase + uint32_t(b) * BN;
          auto ready = [&](int p) {
            if (ok && !tma::wait(&bars.full[b][p], par, err)) ok = false;
          };
          auto product = [&](int pa, int pb, uint32_t d, bool fresh) {
#pragma unroll
            for (int k = 0; k < BK / UK; ++k)
              umma::mma(d, plane_desc<AMN>(st + uint32_t(pa * TILE), k),
                        plane_desc<BMN>(st + uint32_t(pb * TILE), k), ID, (!fresh || k > 0) ? 1u : 0u);
          };
          ready(A3);
          ready(B1);
          if (!ok) break;
          fence_after();
          product(A3, B1, lo, kb == kb0);
          umma::commit(&bars.empty[b][A3]);
          ready(A1);
          ready(B3);
          if (!ok) break;
          fence_after();
          product(A1, B3, lo, false);
          umma::commit(&bars.empty[b][B3]);
          ready(A2);
          ready(B2);
          if (!ok) break;
          fence_after();
          product(A2, B2, lo, false);
          product(A2, B1, lo, false);
          umma::commit(&bars.empty[b][A2]);
          product(A1, B2, lo, false);
          umma::commit(&bars.empty[b][B2]);
          // the epilogue has read out the block this accumulator held before
          if (g >= 2 && !tma::wait(&bars.hie[b], ((g >> 1) - 1u) & 1u, err)) {
            ok = false;
            break;
          }
          fence_after();
          product(A1, B1, hi, true);
          umma::commit(&bars.empty[b][A1]);
          umma::commit(&bars.empty[b][B1]);
          umma::commit(&bars.hif[b]);
        }
      }
      if (!ok) {  // wake the epilogue (it sees the abort) after what was issued
        bars.abort = 1;
        umma::commit(&bars.hif[0]);
        umma::commit(&bars.hif[1]);
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
    int i = 0;
    for (int it = blockIdx.x; it < nitems; it += gridDim.x, ++i) {
      const int s = it / ntiles, t = it - s * ntiles;
      const int nkb = int(int64_t(nk) * (s + 1) / S) - int(int64_t(nk) * s / S);
      bool ready = true;
      float acc[NC];
#pragma unroll
      for (int j = 0; j < NC; ++j) acc[j] = 0.0f;
      auto add_tmem = [&](uint32_t at) {
#pragma unroll
        for (int c = 0; c < NC / 32; ++c) {
          uint32_t r[32];
          ld32(at + uint32_t(c * 32), r);
          umma::wait_ld();
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[c * 32 + j] += __uint_as_float(r[j]);
        }
        fence_before();
        __syncwarp();
      };
      for (int kb = 0; kb < nkb; ++kb, ++g) {
        const int b = int(g & 1u);
        ready = tma::wait(&bars.hif[b], (g >> 1) & 1u, err);
        fence_after();
        // the TMEM loads are warp-wide: the warp decides together
        ready = __all_sync(0xffffffffu, ready && !bars.abort);
        if (!ready) break;
        add_tmem(tmine + uint32_t(b) * BN);
        if (lane == 0) tma::arrive(&bars.hie[b]);
      }
      if (!ready) break;
      add_tmem(tmine + 256u + uint32_t(i & 1) * BN);
      if (lane == 0) tma::arrive(&bars.loe[i & 1]);
      if (S > 1) {
        float* mine = part + int64_t(it) * (BM * BN) + col * BM + row;
#pragma unroll
        for (int j = 0; j < NC; ++j) __stcg(mine + j * BM, acc[j]);
        __threadfence();
        asm volatile("bar.sync 1, %0;" ::"n"(32 * EPI_WARPS) : "memory");
        if (warp == 2 && lane == 0) bars.last = atomicAdd(tickets + t, 1u) == unsigned(S - 1);
        asm volatile("bar.sync 1, %0;" ::"n"(32 * EPI_WARPS) : "memory");
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
      int tm, tn;
      umma::tile_of(t, tiles_m, tiles_n, tm, tn);
      const int64_t m = int64_t(tm) * BM + row;
      if (m < M) store_row<float, E, PS>(e, sl, z, ldz, m, tn * BN + col, N, acc);
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    umma::tmem_dealloc(tbase, 512);
  }
}

// K ranges per tile: the S that minimises waves of work items times their
// length. In K blocks of 64 (about 0.8 us each): an item costs its own blocks
// and about two to fill and drain its pipeline, one more to write and add
// partials when S > 1.
inline int choose_splits(int64_t ntiles, int nk, int sms) {
  int best = 1;
  int64_t cost = 0;
  for (int S = 1; S <= 16 && S <= nk; ++S) {
    const int64_t waves = (ntiles * S + sms - 1) / sms;
    const int64_t c = waves * ((nk + S - 1) / S + 2 + (S > 1 ? 1 : 0));
    if (S == 1 || c < cost) {
      cost = c;
      best = S;
    }
  }
  return best;
}

}  // namespace umma32
}  // namespace fx
