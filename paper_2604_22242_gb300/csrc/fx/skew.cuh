// skew.cuh - tiles of trees with transposed leaves over matrices whose
// columns do not start on 16-byte boundaries (odd row counts, views).
//
// Neither TMA nor an aligned vector tile can address such a matrix, and the
// one-element-wide tile kernel is bound by its loads: at 5003 x 4999 in FP16
// it moves 2 bytes per load instruction and took 114.7 us for Z and s together
// (2180 GB/s of the tree's bytes); the tiles below take 60.6 us (4120 GB/s). But the plain leaves and Z usually share their misalignment:
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
// Vectors that reach over the first or last row are evaluated element by
// element: they exist only in the first and last tile of a column.
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
  static constexpr int SROW = TC + 1;        // odd: rows V apart fall in different banks
  static constexpr int SMEM = NMT * NR * SROW;
};

// Rows row .. row + V - 1 of column c of the plain and broadcast leaves.
template <class LL, int V, class CT, int I = 0>
FX_D void skew_load(Pack<LL, V, CT>& p, const Slots& sl, int64_t row, int64_t c) {
  if constexpr (I < tl_size<LL>::value) {
    using L = typename tl_at<LL, I>::type;
    using TL_ = typename L::elem;
    auto& dst = pget<I>::of(p);
    const SlotView& s = sl.s[L::slot];
    const TL_* base = static_cast<const TL_*>(s.p);
    if constexpr (L::mode == MN) {
      vload(dst, base + row + c * s.ld);
    } else if constexpr (L::mode == MBC) {
#pragma unroll
      for (int j = 0; j < V; ++j) dst.v[j] = sload(base + (row + j) * s.vs);
    } else if constexpr (L::mode == MBR) {
      dst.v[0] = sload(base + c * s.vs);
    }
    skew_load<LL, V, CT, I + 1>(p, sl, row, c);
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
      for (int j = 0; j < VP; ++j) pget<I>::of(p).v[j] = sm[(m * SS::NR + k + j) * SS::SROW + cc];
    }
    skew_fill<SS, VP, I + 1>(p, sm, k, cc);
  }
}

// Piece i of a transposed leaf's tile: D's column r0 - (V - 1) + i / DX,
// elements first .. first + V - 1 (aligned). Returns the tile column of the
// piece's first element, which may be negative; elements outside D stay zero.
template <class SS, class T>
FX_D int skew_piece(Raw<T, SS::V>& w, const SlotView& s, int64_t R, int64_t C, int64_t r0,
                    int64_t c0, int i) {
  constexpr int V = SS::V;
  const int k = i / SS::DX, x = i - k * SS::DX;
  const int64_t r = r0 - (V - 1) + k;
#pragma unroll
  for (int j = 0; j < V; ++j) w.v[j] = T(0.0f);
  if (i >= SS::DN || r < 0 || r >= R) return SS::TC;
  const T* col = static_cast<const T*>(s.p) + r * s.ld;
  const int at = x * V - int(elem_residue<T, V>(col + c0));
  const int64_t first = c0 + at;
  if (first >= 0 && first + V <= C) {
    vload(w, col + first);
  } else {
#pragma unroll
    for (int j = 0; j < V; ++j)
      if (first + j >= 0 && first + j < C) w.v[j] = sload(col + first + j);
  }
  return at;
}

template <class SS, class T, int I = 0>
FX_D void skew_stage(typename SS::CT* sm, const Slots& sl, int64_t R, int64_t C, int64_t r0,
                     int64_t c0, bool& fresh) {
  using LL = typename SS::LL;
  using CT = typename SS::CT;
  if constexpr (I < tl_size<LL>::value) {
    using L = typename tl_at<LL, I>::type;
    if constexpr (L::mode == MT) {
      constexpr int m = mt_rank<LL, I>();
      Raw<T, SS::V> w[SS::DP];
      int at[SS::DP];
#pragma unroll
      for (int q = 0; q < SS::DP; ++q)
        at[q] = skew_piece<SS, T>(w[q], sl.s[L::slot], R, C, r0, c0, int(threadIdx.x) + q * SS::NT);
      if (!fresh) __syncthreads();  // the previous tile's readers are done with sm
      fresh = true;
#pragma unroll
      for (int q = 0; q < SS::DP; ++q) {
        const int i = int(threadIdx.x) + q * SS::NT;
        CT* row = sm + (m * SS::NR + i / SS::DX) * SS::SROW;
        if (i < SS::DN) {
#pragma unroll
          for (int j = 0; j < SS::V; ++j) {
            const int cc = at[q] + j;
            if (cc >= 0 && cc < SS::TC) row[cc] = to_compute<CT>(w[q].v[j]);
          }
        }
      }
    }
    skew_stage<SS, T, I + 1>(sm, sl, R, C, r0, c0, fresh);
  }
}

template <class E, class EpiV, class Epi1, class T, int V, int TR, int TC, int NT>
__global__ void __launch_bounds__(NT) k_tile_skew(const E e, const Slots sl, const int64_t R,
                                                  const int64_t C, const EpiV ev, const Epi1 e1,
                                                  const RedArgs red, const uint32_t sbase,
                                                  const uint32_t sld) {
  using SS = SkewShape<E, T, V, TR, TC, NT>;
  using LL = typename SS::LL;
  using CT = typename SS::CT;
  static_assert(SS::NMT > 0, "trees with a transposed leaf");
  __shared__ CT sm[SS::SMEM];
  typename EpiV::State st;
  st.init();
  constexpr bool one_state = std::is_same<typename EpiV::State, typename Epi1::State>::value;
  static_assert(one_state || !EpiV::reduces, "single elements join the same running sum");
  typename Epi1::State none;
  auto& st1 = [&]() -> typename Epi1::State& {
    if constexpr (one_state) return st;
    else return none;
  }();
  const int64_t tiles_r = (R + V - 1 + TR - 1) / TR, tiles_c = (C + TC - 1) / TC;
  const int64_t ntiles = tiles_r * tiles_c;
  const int tx = threadIdx.x % SS::TX, ty = threadIdx.x / SS::TX;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    int64_t tr, tc;
    tile_coords(t, tiles_r, tiles_c, tr, tc);
    const int64_t r0 = tr * TR, c0 = tc * TC;
    Pack<LL, V, CT> p[SS::P];
#pragma unroll
    for (int q = 0; q < SS::P; ++q) {
      const int64_t c = c0 + ty + q * SS::TY;
      const int sk = int((sbase + uint32_t(c) * sld) & uint32_t(V - 1));
      const int64_t row = r0 - sk + tx * V;
      if (c < C && row >= 0 && row + V <= R) skew_load(p[q], sl, row, c);
    }
    bool fresh = false;
    skew_stage<SS, T>(sm, sl, R, C, r0, c0, fresh);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < SS::P; ++q) {
      const int cc = ty + q * SS::TY;
      const int64_t c = c0 + cc;
      if (c >= C) continue;
      const int sk = int((sbase + uint32_t(c) * sld) & uint32_t(V - 1));
      const int64_t row = r0 - sk + tx * V;
      const int k = tx * V - sk + V - 1;  // staged row of lane 0
      if (row >= 0 && row + V <= R) {
        skew_fill<SS, V>(p[q], sm, k, cc);
        CT v[V];
        eval_lanes<V>(e, p[q], v);
        epi_put(ev, st, row + c * ev.ldz, v, p[q], V);
      } else {
#pragma unroll 1
        for (int j = 0; j < V; ++j) {
          if (row + j < 0 || row + j >= R) continue;
          Pack<LL, 1, CT> p1;
          load_rc(p1, sl, row + j, c, 1);
          skew_fill<SS, 1>(p1, sm, k + j, cc);
          CT v1[1];
          eval_lanes<1>(e, p1, v1);
          epi_put(e1, st1, row + j + c * e1.ldz, v1, p1, 1);
        }
      }
    }
  }
  if constexpr (EpiV::reduces) finish_full_reduce<CT, EpiV::sqrt_result>(st, red);
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

// Can k_tile_skew take these operands? (z null: a tree that stores nothing)
template <class LL, class T, int V>
bool skew_ok(const Binding* b, const void* z, int64_t ldz, uint32_t& sbase, uint32_t& sld) {
  int first = -1;
  if (!skew_leaves<LL, T, V>(b, first, sbase, sld) || first < 0) return false;
  return !z || (elem_residue<T, V>(z) == sbase && (uint32_t(ldz) & uint32_t(V - 1)) == sld);
}

}  // namespace fx
