// skew.cuh - tiles of trees with transposed leaves over matrices whose
// columns do not start on 16-byte boundaries (odd row counts, views).
//
// Neither TMA nor an aligned vector tile can address such a matrix, and the
// one-element-wide tile kernel is bound by its loads: at 5003 x 4999 in FP16
// it moves 2 bytes per load instruction and took 114.7 us for Z and s together
// (2180 GB/s of the tree's bytes); the tiles below take 59.5 us (4200 GB/s). But the plain leaves and Z usually share their misalignment:
// with equal base residues and leading dimensions equal modulo V (V elements
// = 16 bytes), element (r, c) of all of them sits at the same offset in its
// 16-byte line. A tile here takes, in column c, the rows r0 - s(c) ..
// r0 - s(c) + TR - 1, s(c) = (sbase + c sld) mod V, so that every V-row
// vector of every plain leaf and of Z is one aligned 16-byte access.
//
// A transposed leaf D is read along its own columns in aligned 16-byte
// pieces, each column with its own misalignment (one more piece than an
// aligned tile has), and staged in shared memory as S[row][column] for the
// TR + V - 1 output rows that the shifts can reach.
//
// Vectors that reach over the first or last row load and store their
// elements inside one by one. Tiles away from the matrix's edges run without
// any of the checks.
#pragma once

#include "kernels.cuh"
#include "runtime.hpp"

namespace fx {

// Misalignment in elements of address p (0 .. V - 1).
template <class T, int V> FX_HD uint32_t elem_residue(const void* p) {
  return uint32_t(reinterpret_cast<uintptr_t>(p) / sizeof(T)) & uint32_t(V - 1);
}

template <class E, class T, int V_, int TR_, int TC_, int NT_> struct SkewShape {
  using LL = leaves_t<E>;
  using CT = ct_of<E>;
  static constexpr int V = V_, TR = TR_, TC = TC_, NT = NT_;
  static constexpr int TX = TR / V, TY = NT / TX, P = TC / TY;
  static_assert(TX * V == TR && TX * TY == NT && P * TY == TC, "bad tile shape");
  static constexpr int NR = TR + V - 1;      // staged output rows (D's columns)
  static constexpr int DX = TC / V + 1;      // 16-byte pieces per column of D
  static constexpr int DN = NR * DX;         // pieces per transposed leaf
  static constexpr int DP = (DN + NT - 1) / NT;
  static constexpr int NMT = count_mt<LL>();
  // a staged row: V columns of margin on both sides, so that whole pieces are
  // stored without a check per element; odd, so that rows fall in different banks
  static constexpr int SROW = TC + 2 * V + 1;
  static constexpr int SMEM = NMT > 0 ? NMT * NR * SROW : 1;
};

// Where a tile lies and how its columns are shifted. Tiles start at multiples
// of V in both directions, so the shift of a column, and the misalignment of
// a transposed leaf's column, depend on its place in the tile alone. Extents
// are below 2^31 and leading dimensions below 2^25 (the host checks): offsets
// inside a tile are 32-bit.
struct SkewPlace {
  int R, C, r0, c0;
  uint32_t sbase, sld;
};
template <int V> FX_D int col_shift(const SkewPlace& t, int cc) {
  return int((t.sbase + uint32_t(cc) * t.sld) & uint32_t(V - 1));
}
// Operands of one matrix, from the kernel's arguments.
struct ArgSlots {
  const Slots& sl;
  FX_D SlotView operator()(int slot) const { return sl.s[slot]; }
};

// Rows r0 + rel .. r0 + rel + V - 1 of tile column cc of the plain and
// broadcast leaves; get(slot) gives a leaf's SlotView. ALL: the whole vector
// is inside the matrix, else rows r0 + rel + lo .. r0 + rel + hi - 1 are.
template <bool ALL, class LL, int V, class CT, class Get, int I = 0>
FX_D void skew_load(Pack<LL, V, CT>& p, const Get& get, const SkewPlace& t, int rel, int cc, int lo,
                    int hi) {
  if constexpr (I < tl_size<LL>::value) {
    using L = typename tl_at<LL, I>::type;
    using TL_ = typename L::elem;
    auto& dst = pget<I>::of(p);
    if constexpr (L::mode != MT) {
      const SlotView s = get(L::slot);
      const TL_* base = static_cast<const TL_*>(s.p);
      if constexpr (L::mode == MN) {
        const TL_* q = base + (t.r0 + int64_t(t.c0) * s.ld) + (rel + cc * int(s.ld));
        if constexpr (ALL) {
          vload(dst, q);
        } else {
#pragma unroll
          for (int j = 0; j < V; ++j) dst.v[j] = j >= lo && j < hi ? sload(q + j) : TL_(0.0f);
        }
      } else if constexpr (L::mode == MBC) {
#pragma unroll
        for (int j = 0; j < V; ++j)
          dst.v[j] = ALL || (j >= lo && j < hi) ? sload(base + int64_t(t.r0 + rel + j) * s.vs) : TL_(0.0f);
      } else {
        dst.v[0] = sload(base + int64_t(t.c0 + cc) * s.vs);
      }
    }
    skew_load<ALL, LL, V, CT, Get, I + 1>(p, get, t, rel, cc, lo, hi);
  }
}

// The transposed leaves' values from the staged rows: lane j of the vector
// is staged row k + j, tile column cc.
template <class SS, int VP, int I = 0>
FX_D void skew_fill(Pack<typename SS::LL, VP, typename SS::CT>& p, const typename SS::CT* sm, int k,
                    int cc) {
  using LL = typename SS::LL;
  if constexpr (I < tl_size<LL>::value) {
    using L = typename tl_at<LL, I>::type;
    if constexpr (L::mode == MT) {
      constexpr int m = mt_rank<LL, I>();
#pragma unroll
      for (int j = 0; j < VP; ++j) pget<I>::of(p).v[j] = sm[(m * SS::NR + k + j) * SS::SROW + SS::V + cc];
    }
    skew_fill<SS, VP, I + 1>(p, sm, k, cc);
  }
}

// Piece i of a transposed leaf's tile: 16 aligned bytes of D's column
// r0 - (V - 1) + i / DX. Returns the tile column of the piece's first
// element, which may be negative; elements outside D stay zero (IN: the tile
// and its margins are inside).
template <class SS, class T, bool IN>
FX_D int skew_piece(Raw<T, SS::V>& w, const SlotView& s, const SkewPlace& t, int i) {
  constexpr int V = SS::V;
  const int k = i / SS::DX, x = i - k * SS::DX, dr = k - (V - 1);
  const T* tile = static_cast<const T*>(s.p) + (t.c0 + int64_t(t.r0) * s.ld);
  const int at = x * V - int((elem_residue<T, V>(tile) + uint32_t(dr) * uint32_t(s.ld)) & uint32_t(V - 1));
  const T* src = tile + (at + dr * int(s.ld));
  if constexpr (IN) {
    if (i < SS::DN) vload(w, src);
  } else {
#pragma unroll
    for (int j = 0; j < V; ++j) w.v[j] = T(0.0f);
    if (i < SS::DN && uint32_t(t.r0 + dr) < uint32_t(t.R)) {
      const int first = t.c0 + at;
      if (first >= 0 && first + V <= t.C) {
        vload(w, src);
      } else {
#pragma unroll
        for (int j = 0; j < V; ++j)
          if (first + j >= 0 && first + j < t.C) w.v[j] = sload(src + j);
      }
    }
  }
  return at;
}

// Loads and stages the transposed leaves' tiles. between() runs after the
// barrier that ends the previous tile's reads of sm.
template <class SS, class T, bool IN, class Get, class B, int I = 0>
FX_D void skew_stage(typename SS::CT* sm, const Get& get, const SkewPlace& t, const B& between,
                     bool joined = false) {
  using LL = typename SS::LL;
  using CT = typename SS::CT;
  if constexpr (I < tl_size<LL>::value) {
    using L = typename tl_at<LL, I>::type;
    if constexpr (L::mode == MT) {
      constexpr int m = mt_rank<LL, I>();
      const SlotView s = get(L::slot);
      Raw<T, SS::V> w[SS::DP];
      int at[SS::DP];
#pragma unroll
      for (int q = 0; q < SS::DP; ++q)
        at[q] = skew_piece<SS, T, IN>(w[q], s, t, int(threadIdx.x) + q * SS::NT);
      if (!joined) {
        __syncthreads();
        between();
        joined = true;
      }
#pragma unroll
      for (int q = 0; q < SS::DP; ++q) {
        const int i = int(threadIdx.x) + q * SS::NT;
        CT* row = sm + (m * SS::NR + i / SS::DX) * SS::SROW;
        if (i < SS::DN) {
#pragma unroll
          for (int j = 0; j < SS::V; ++j) row[SS::V + at[q] + j] = to_compute<CT>(w[q].v[j]);
        }
      }
    }
    skew_stage<SS, T, IN, Get, B, I + 1>(sm, get, t, between, joined);
  } else if (!joined) {
    __syncthreads();
    between();
  }
}

// One tile: out.full(pack, values, rel, cc) for a vector inside the matrix,
// out.part(pack, values, rel, cc, lo, hi) for one whose lanes lo .. hi - 1 are.
// IN: the tile, shifted by up to V - 1 rows, and the transposed leaves' pieces
// are inside the matrix.
template <class SS, class T, bool IN, class E, class Get, class B, class Out>
FX_D void skew_tile_of(const E& e, const Get& get, const SkewPlace& t, typename SS::CT* sm,
                       const B& between, const Out& out) {
  using LL = typename SS::LL;
  using CT = typename SS::CT;
  constexpr int V = SS::V;
  const int tx = threadIdx.x % SS::TX, ty = threadIdx.x / SS::TX;
  Pack<LL, V, CT> p[SS::P];
  int lo[SS::P], hi[SS::P];  // lanes inside (none: lo >= hi)
#pragma unroll
  for (int q = 0; q < SS::P; ++q) {
    const int cc = ty + q * SS::TY, rel = tx * V - col_shift<V>(t, cc);
    if constexpr (IN) {
      skew_load<true>(p[q], get, t, rel, cc, 0, V);
    } else {
      const int row = t.r0 + rel;
      lo[q] = row < 0 ? -row : 0;
      hi[q] = t.c0 + cc >= t.C ? 0 : (t.R - row < V ? t.R - row : V);
      if (lo[q] == 0 && hi[q] == V) skew_load<true>(p[q], get, t, rel, cc, 0, V);
      else if (lo[q] < hi[q]) skew_load<false>(p[q], get, t, rel, cc, lo[q], hi[q]);
    }
  }
  skew_stage<SS, T, IN>(sm, get, t, between);
  __syncthreads();
#pragma unroll
  for (int q = 0; q < SS::P; ++q) {
    const int cc = ty + q * SS::TY, rel = tx * V - col_shift<V>(t, cc);
    if (!IN && lo[q] >= hi[q]) continue;
    skew_fill<SS, V>(p[q], sm, rel + V - 1, cc);
    CT v[V];
    eval_lanes<V>(e, p[q], v);
    if (IN || (lo[q] == 0 && hi[q] == V)) out.full(p[q], v, rel, cc);
    else out.part(p[q], v, rel, cc, lo[q], hi[q]);
  }
}
template <class SS, class T, class E, class Get, class B, class Out>
FX_D void skew_tile(const E& e, const Get& get, const SkewPlace& t, typename SS::CT* sm,
                    const B& between, const Out& out) {
  constexpr int V = SS::V;
  const bool in = t.r0 >= V && t.r0 + SS::TR <= t.R && t.c0 >= V && t.c0 + SS::TC + V <= t.C;
  if (in) skew_tile_of<SS, T, true>(e, get, t, sm, between, out);
  else skew_tile_of<SS, T, false>(e, get, t, sm, between, out);
}

// Threads per block, and blocks per SM that the register budget is cut for. 4-
// and 8-byte types have twice the vectors per tile; Z and s at 5003 x 4999 FP32:
// 85.6 us with two blocks of 256 threads, 89.9 with two of 512; in BF16 59.3
// with three of 256, 64.6 with two.
constexpr int skew_threads() { return 256; }
template <class T> constexpr int skew_blocks() { return sizeof(T) == 2 ? 3 : 2; }

struct Nothing {
  FX_D void operator()() const {}
};
// Brings the leaves' part of tile t towards L2, a 128-byte line per entry:
// entries threadIdx.x, + NT, ... of each leaf's columns. The next tile is
// known while the current one loads, and only registers limit how early its
// loads could be issued; its lines in L2 leave them the shorter wait. For the
// batch (4096 matrices FP32: 2665 us without, 2372 with); one large matrix,
// whose tiles the other blocks bring in anyway, is slower with it (Z and s at
// 5003 x 4999 FP32 96.5 against 85.6 us).
template <class SS, class T, class Get, int I = 0>
FX_D void skew_prefetch(const Get& get, const SkewPlace& t) {
  using LL = typename SS::LL;
  if constexpr (I < tl_size<LL>::value) {
    using L = typename tl_at<LL, I>::type;
    if constexpr (L::mode == MN || L::mode == MT) {
      constexpr bool tr = L::mode == MT;
      constexpr int LE = 128 / int(sizeof(T));                  // elements of a line
      constexpr int LPC = ((tr ? SS::TC : SS::TR) + LE - 1) / LE;  // lines of a column
      constexpr int N = (tr ? SS::TR : SS::TC) * LPC;
      const SlotView s = get(L::slot);
      const int R = tr ? t.C : t.R, C = tr ? t.R : t.C, r0 = tr ? t.c0 : t.r0, c0 = tr ? t.r0 : t.c0;
#pragma unroll
      for (int q = 0; q < (N + SS::NT - 1) / SS::NT; ++q) {
        const int i = int(threadIdx.x) + q * SS::NT;
        const int r = r0 + i % LPC * LE, c = c0 + i / LPC;
        if (i < N && r < R && c < C)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const T*>(s.p) + r + int64_t(c) * s.ld));
      }
    }
    skew_prefetch<SS, T, Get, I + 1>(get, t);
  }
}
// Hands a tile's values to the epilogue. `at`: the tile's first element in Z.
template <class T, class Epi> struct SkewEpi {
  const Epi& epi;
  typename Epi::State& st;
  int64_t at;
  template <class P, class CT, int V> FX_D void full(const P& p, const CT (&v)[V], int rel, int cc) const {
    epi_put(epi, st, at + (rel + cc * int(epi.ldz)), v, p, V);
  }
  template <class LL, class CT, int V>
  FX_D void part(const Pack<LL, V, CT>& p, const CT (&v)[V], int rel, int cc, int lo, int hi) const {
    const int64_t off = at + (rel + cc * int(epi.ldz));
#pragma unroll
    for (int j = 0; j < V; ++j) {
      if (j < lo || j >= hi) continue;
      if constexpr (Epi::stores) sstore(epi.z + off + j, narrow_to<T>::from(v[j]));
      if constexpr (Epi::side_tree) {
        Ctx<LL, V, CT> cx{p, j};
        st.add(epi.side.ev(cx));
      } else if constexpr (Epi::reduces) {
        st.add(Epi::sqrt_result ? v[j] * v[j] : v[j]);
      }
    }
  }
};

template <class E, class Epi, class T, int V, int TR, int TC, int NT>
__global__ void __launch_bounds__(NT, skew_blocks<T>()) k_tile_skew(const E e, const Slots sl, const int64_t R,
                                                  const int64_t C, const Epi epi, const RedArgs red,
                                                  const uint32_t sbase, const uint32_t sld,
                                                  const int64_t tiles_r) {
  using SS = SkewShape<E, T, V, TR, TC, NT>;
  using CT = typename SS::CT;
  static_assert(SS::NMT > 0, "trees with a transposed leaf");
  __shared__ CT sm[SS::SMEM];
  typename Epi::State st;
  st.init();
  const int64_t tiles_c = (C + TC - 1) / TC;
  const int64_t ntiles = tiles_r * tiles_c;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    int64_t tr, tc;
    tile_coords(t, tiles_r, tiles_c, tr, tc);
    skew_tile<SS, T>(e, ArgSlots{sl}, SkewPlace{int(R), int(C), int(tr * TR), int(tc * TC), sbase, sld},
                     sm, Nothing{}, SkewEpi<T, Epi>{epi, st, tr * TR + tc * TC * epi.ldz});
  }
  if constexpr (Epi::reduces) finish_full_reduce<CT, Epi::sqrt_result>(st, red);
}

// ---------------------------------------------------------------- host side

// Every plain leaf has residue (base, ld mod V) = (sbase, sld); first < 0
// until one is met.
template <class LL, class T, int V, int I = 0>
bool skew_leaves(const Binding* b, int& first, uint32_t& sbase, uint32_t& sld) {
  if constexpr (I < tl_size<LL>::value) {
    using L = typename tl_at<LL, I>::type;
    if constexpr (L::mode == MN) {
      const Binding& x = b[L::slot];
      const uint32_t base = elem_residue<T, V>(x.p), ld = uint32_t(x.ld) & uint32_t(V - 1);
      if (first < 0) {
        first = L::slot;
        sbase = base;
        sld = ld;
      } else if (base != sbase || ld != sld) {
        return false;
      }
    }
    return skew_leaves<LL, T, V, I + 1>(b, first, sbase, sld);
  }
  return true;
}

// Rows and columns that the tiles can count in 32 bits: the last tile begins
// up to a shift beyond the last row, and its end and the rows of its vectors
// are computed too.
constexpr int64_t kSkewExtent = (int64_t(1) << 31) - 128;
inline bool skew_extent(int64_t R, int64_t C) { return R < kSkewExtent && C < kSkewExtent; }

// Offsets inside a tile are 32-bit: leading dimensions below 2^25.
constexpr int64_t kSkewLd = int64_t(1) << 25;
template <class LL, int I = 0> bool skew_lds(const Binding* b) {
  if constexpr (I < tl_size<LL>::value) {
    using L = typename tl_at<LL, I>::type;
    if ((L::mode == MN || L::mode == MT) && b[L::slot].ld >= kSkewLd) return false;
    return skew_lds<LL, I + 1>(b);
  }
  return true;
}

// Do the plain leaves and Z share their misalignment? (z null: nothing stored)
template <class LL, class T, int V>
bool skew_ok(const Binding* b, const void* z, int64_t ldz, uint32_t& sbase, uint32_t& sld) {
  int first = -1;
  if (!skew_lds<LL>(b) || (z && ldz >= kSkewLd)) return false;
  if (!skew_leaves<LL, T, V>(b, first, sbase, sld) || first < 0) return false;
  return !z || (elem_residue<T, V>(z) == sbase && (uint32_t(ldz) & uint32_t(V - 1)) == sld);
}

// The largest shift of any of the first C columns.
template <int V> int max_shift(uint32_t sbase, uint32_t sld, int64_t C) {
  uint32_t m = 0;
  for (int64_t c = 0; c < C && c < V; ++c) {
    const uint32_t s = (sbase + uint32_t(c) * sld) & uint32_t(V - 1);
    m = s > m ? s : m;
  }
  return int(m);
}

}  // namespace fx
