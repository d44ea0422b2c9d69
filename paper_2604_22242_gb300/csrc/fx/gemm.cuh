// gemm.cuh - matrix products inside a tree: the fusion boundary.
//
// A matrix product cannot be computed one output element at a time from one
// element of each operand, so the planner treats it as a boundary (Sec. 5:
// the fused kernel covers the element-wise part of an expression): every
// product node, innermost first, is computed by a library GEMM (cuBLAS,
// FP32/FP64 arithmetic, BF16/FP16 operands with FP32 accumulation) into a
// temporary matrix of the storage type, the product node is replaced by a
// plain leaf bound to that temporary, and the rest of the tree runs on the
// fused path as usual. Two roots need no second pass: a bare product and a
// scalar times a product (Fig. 1's Z = 2 X Y^T), whose scalar becomes the
// GEMM's alpha and whose output is written straight into Z. Trees with one
// product of matrix leaves and an element-wise remainder run on the tensor
// cores in one kernel instead (umma.cuh for BF16 and FP16, umma32.cuh for
// FP32), where their sizes and operands allow it.
//
// Product operands must be matrix leaves, plain or transposed (a transpose
// becomes the GEMM's operand op), or products themselves (the paper's
// chain Z = A * B * C * D).
#pragma once

#include <initializer_list>

#include <cublas_v2.h>

#include "umma.cuh"
#include "umma32.cuh"
#include "unfused.cuh"

namespace fx {

// ---------------------------------------------------------------- lifting

// Lift<E, T, S>: E with its product nodes replaced, in post-order, by plain
// leaves of storage type T at slots S, S+1, ...; count = number replaced.
template <class E, class T, int S> struct Lift {
  using type = E;
  static constexpr int count = 0;
  static FX_HD type make(const E& e) { return e; }
};
template <class Op, class L, class R, class T, int S> struct Lift<Bin<Op, L, R>, T, S> {
  using LA = Lift<L, T, S>;
  using RA = Lift<R, T, S + LA::count>;
  using type = Bin<Op, typename LA::type, typename RA::type>;
  static constexpr int count = LA::count + RA::count;
  static FX_HD type make(const Bin<Op, L, R>& e) { return {{}, LA::make(e.l), RA::make(e.r)}; }
};
template <class Op, class E, class T, int S> struct Lift<Un<Op, E>, T, S> {
  using A = Lift<E, T, S>;
  using type = Un<Op, typename A::type>;
  static constexpr int count = A::count;
  static FX_HD type make(const Un<Op, E>& e) { return {{}, A::make(e.e)}; }
};
template <class Op, class E, class T, int S> struct Lift<SL<Op, E>, T, S> {
  using A = Lift<E, T, S>;
  using type = SL<Op, typename A::type>;
  static constexpr int count = A::count;
  static FX_HD type make(const SL<Op, E>& e) { return {{}, e.s, A::make(e.e)}; }
};
template <class Op, class E, class T, int S> struct Lift<SR<Op, E>, T, S> {
  using A = Lift<E, T, S>;
  using type = SR<Op, typename A::type>;
  static constexpr int count = A::count;
  static FX_HD type make(const SR<Op, E>& e) { return {{}, A::make(e.e), e.s}; }
};
template <class L, class R, class T, int S> struct Lift<Prod<L, R>, T, S> {
  using LA = Lift<L, T, S>;
  using RA = Lift<R, T, S + LA::count>;
  static constexpr int slot = S + LA::count + RA::count;
  using type = Leaf<slot, T, MN>;
  static constexpr int count = LA::count + RA::count + 1;
  static FX_HD type make(const Prod<L, R>&) { return {}; }
};
template <class E, class T, int S> struct Lift<Accu<E>, T, S> {
  using A = Lift<E, T, S>;
  using type = Accu<typename A::type>;
  static constexpr int count = A::count;
  static FX_HD type make(const Accu<E>& e) { return {{}, A::make(e.e)}; }
};
template <class E, class T, int S> struct Lift<Norm2<E>, T, S> {
  using A = Lift<E, T, S>;
  using type = Norm2<typename A::type>;
  static constexpr int count = A::count;
  static FX_HD type make(const Norm2<E>& e) { return {{}, A::make(e.e)}; }
};
template <class E, int D, class T, int S> struct Lift<SumDim<E, D>, T, S> {
  using A = Lift<E, T, S>;
  using type = SumDim<typename A::type, D>;
  static constexpr int count = A::count;
  static FX_HD type make(const SumDim<E, D>& e) { return {{}, A::make(e.e)}; }
};
template <class E, int D, class T, int S> struct Lift<MaxDim<E, D>, T, S> {
  using A = Lift<E, T, S>;
  using type = MaxDim<typename A::type, D>;
  static constexpr int count = A::count;
  static FX_HD type make(const MaxDim<E, D>& e) { return {{}, A::make(e.e)}; }
};

template <class E> struct has_prod_any { static constexpr bool value = has_prod_v<E>; };
template <class E> struct has_prod_any<Accu<E>> { static constexpr bool value = has_prod_v<E>; };
template <class E> struct has_prod_any<Norm2<E>> { static constexpr bool value = has_prod_v<E>; };
template <class E, int D> struct has_prod_any<SumDim<E, D>> { static constexpr bool value = has_prod_v<E>; };
template <class E, int D> struct has_prod_any<MaxDim<E, D>> { static constexpr bool value = has_prod_v<E>; };

// ---------------------------------------------------------------- cuBLAS

inline fx_status blas_fail(cublasStatus_t s, const char* what) {
  return fail(FX_E_CUDA, "%s: cuBLAS status %d", what, int(s));
}

// One handle per thread and device, created on first use.
inline fx_status blas_handle(cublasHandle_t* out) {
  struct Handles {
    cublasHandle_t h[64] = {};
    ~Handles() {
      for (auto& x : h)
        if (x) cublasDestroy(x);
    }
  };
  static thread_local Handles hs;
  int dev = 0;
  FX_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(FX_E_UNSUPPORTED, "device %d", dev);
  if (!hs.h[dev]) {
    const cublasStatus_t s = cublasCreate(&hs.h[dev]);
    if (s != CUBLAS_STATUS_SUCCESS) return blas_fail(s, "cublasCreate");
    cublasSetMathMode(hs.h[dev], CUBLAS_DEFAULT_MATH);  // full FP32, no TF32
  }
  *out = hs.h[dev];
  return FX_OK;
}

template <class T> struct BlasType;
template <> struct BlasType<float> {
  static constexpr cudaDataType data = CUDA_R_32F;
  static constexpr cublasComputeType_t compute = CUBLAS_COMPUTE_32F;
  using scale = float;
};
template <> struct BlasType<double> {
  static constexpr cudaDataType data = CUDA_R_64F;
  static constexpr cublasComputeType_t compute = CUBLAS_COMPUTE_64F;
  using scale = double;
};
template <> struct BlasType<bf16> {
  static constexpr cudaDataType data = CUDA_R_16BF;
  static constexpr cublasComputeType_t compute = CUBLAS_COMPUTE_32F;
  using scale = float;
};
template <> struct BlasType<f16> {
  static constexpr cudaDataType data = CUDA_R_16F;
  static constexpr cublasComputeType_t compute = CUBLAS_COMPUTE_32F;
  using scale = float;
};

// A product operand after lifting: a plain or transposed matrix leaf.
template <class O> struct Operand;
template <int K, class T, int M> struct Operand<Leaf<K, T, M>> {
  static_assert(M == MN || M == MT, "a product operand is a matrix, plain or transposed");
  static constexpr int slot = K;
  static constexpr bool trans = M == MT;
};

// C (m x n, leading dimension ldc) = alpha * op(A) * op(B) for lifted
// operand leaves LA, LB bound in b.
template <class T, class LA, class LB>
fx_status gemm_into(const Binding* b, void* c, int64_t ldc, int64_t m_expect, int64_t n_expect,
                    double alpha, cudaStream_t st) {
  using OA = Operand<LA>;
  using OB = Operand<LB>;
  const Binding& a = b[OA::slot];
  const Binding& bb = b[OB::slot];
  const int64_t m = OA::trans ? a.cols : a.rows, ka = OA::trans ? a.rows : a.cols;
  const int64_t kb = OB::trans ? bb.cols : bb.rows, n = OB::trans ? bb.rows : bb.cols;
  if (ka != kb) return fail(FX_E_SHAPE, "matrix product: inner sizes %lld and %lld differ",
                            (long long)ka, (long long)kb);
  if (m != m_expect || n != n_expect)
    return fail(FX_E_SHAPE, "matrix product is %lld x %lld, expected %lld x %lld", (long long)m,
                (long long)n, (long long)m_expect, (long long)n_expect);
  const int64_t lim = int64_t(1) << 31;
  if (m >= lim || n >= lim || ka >= lim || a.ld >= lim || bb.ld >= lim || ldc >= lim)
    return fail(FX_E_SHAPE, "matrix product too large for a 32-bit GEMM");
  if (m == 0 || n == 0) return FX_OK;
  cublasHandle_t h;
  FX_TRY(blas_handle(&h));
  cublasStatus_t s = cublasSetStream(h, st);
  if (s != CUBLAS_STATUS_SUCCESS) return blas_fail(s, "cublasSetStream");
  using BT = BlasType<T>;
  const typename BT::scale al = typename BT::scale(alpha), be = typename BT::scale(0);
  s = cublasGemmEx(h, OA::trans ? CUBLAS_OP_T : CUBLAS_OP_N, OB::trans ? CUBLAS_OP_T : CUBLAS_OP_N,
                   int(m), int(n), int(ka), &al, a.p, BT::data, int(a.ld > 0 ? a.ld : 1), bb.p,
                   BT::data, int(bb.ld > 0 ? bb.ld : 1), &be, c, BT::data, int(ldc > 0 ? ldc : 1),
                   BT::compute, CUBLAS_GEMM_DEFAULT);
  if (s != CUBLAS_STATUS_SUCCESS) return blas_fail(s, "cublasGemmEx");
  return FX_OK;
}

// Rows and columns of a lifted product operand.
template <class L> void operand_shape(const Binding* b, int64_t& r, int64_t& c) {
  using O = Operand<L>;
  const Binding& x = b[O::slot];
  r = O::trans ? x.cols : x.rows;
  c = O::trans ? x.rows : x.cols;
}

// Computes every product of E (normalised, unlifted), innermost first,
// into temporaries bound at slots S, S+1, ... of b (the order Lift uses),
// carved from `base` at running byte offset `off`. With dry set, only the
// bindings' shapes and offsets are set (to size the workspace).
template <class T, int S, class E> struct Prods {
  static fx_status run(Binding*, const E&, char*, size_t&, bool, cudaStream_t) { return FX_OK; }
};
template <class T, int S, class Op, class L, class R> struct Prods<T, S, Bin<Op, L, R>> {
  static fx_status run(Binding* b, const Bin<Op, L, R>& e, char* base, size_t& off, bool dry,
                       cudaStream_t st) {
    FX_TRY((Prods<T, S, L>::run(b, e.l, base, off, dry, st)));
    return Prods<T, S + Lift<L, T, S>::count, R>::run(b, e.r, base, off, dry, st);
  }
};
template <class T, int S, class Op, class E> struct Prods<T, S, Un<Op, E>> {
  static fx_status run(Binding* b, const Un<Op, E>& e, char* base, size_t& off, bool dry,
                       cudaStream_t st) {
    return Prods<T, S, E>::run(b, e.e, base, off, dry, st);
  }
};
template <class T, int S, class Op, class E> struct Prods<T, S, SL<Op, E>> {
  static fx_status run(Binding* b, const SL<Op, E>& e, char* base, size_t& off, bool dry,
                       cudaStream_t st) {
    return Prods<T, S, E>::run(b, e.e, base, off, dry, st);
  }
};
template <class T, int S, class Op, class E> struct Prods<T, S, SR<Op, E>> {
  static fx_status run(Binding* b, const SR<Op, E>& e, char* base, size_t& off, bool dry,
                       cudaStream_t st) {
    return Prods<T, S, E>::run(b, e.e, base, off, dry, st);
  }
};
template <class T, int S, class L, class R> struct Prods<T, S, Prod<L, R>> {
  static fx_status run(Binding* b, const Prod<L, R>& e, char* base, size_t& off, bool dry,
                       cudaStream_t st) {
    using LA = Lift<L, T, S>;
    using RA = Lift<R, T, S + LA::count>;
    FX_TRY((Prods<T, S, L>::run(b, e.l, base, off, dry, st)));
    FX_TRY((Prods<T, S + LA::count, R>::run(b, e.r, base, off, dry, st)));
    int64_t m, k1, k2, n;
    operand_shape<typename LA::type>(b, m, k1);
    operand_shape<typename RA::type>(b, k2, n);
    if (k1 != k2)
      return fail(FX_E_SHAPE, "matrix product: inner sizes %lld and %lld differ", (long long)k1,
                  (long long)k2);
    Binding& out = b[Lift<Prod<L, R>, T, S>::slot];
    out.p = base + off;
    out.rows = m;
    out.cols = n;
    out.ld = m > 0 ? m : 1;
    out.bound = true;
    off += ((size_t(m) * size_t(n) * sizeof(T)) + 255) & ~size_t(255);
    if (dry) return FX_OK;
    return gemm_into<T, typename LA::type, typename RA::type>(b, out.p, out.ld, m, n, 1.0, st);
  }
};

}  // namespace fx

namespace fx {

// Roots whose products need no second pass: a product, or a scalar times a
// product (the scalar becomes the GEMM's alpha).
template <class Root> struct ScaledProd {
  static constexpr bool value = false;
};
template <class L, class R> struct ScaledProd<Prod<L, R>> {
  static constexpr bool value = true;
  using P = Prod<L, R>;
  static double scale(const P&) { return 1.0; }
  static const P& prod(const P& p) { return p; }
};
template <class L, class R> struct ScaledProd<SL<OpMul, Prod<L, R>>> {
  static constexpr bool value = true;
  using P = Prod<L, R>;
  static double scale(const SL<OpMul, P>& e) { return e.s; }
  static const P& prod(const SL<OpMul, P>& e) { return e.e; }
};

// ---------------------------------------------------------------- tcgen05 path

// Trees the tensor-core kernels take: BF16, FP16 or FP32 storage, one matrix
// product of two matrix leaves (plain or transposed), and an element-wise
// remainder whose other leaves are plain matrices of the storage type.
template <class T, int NIN, class Root> struct umma_ok {
  static constexpr bool value = [] {
    if constexpr (std::is_same<T, double>::value) {
      return false;
    } else if constexpr (root_of<Root>::kind != FX_KIND_ELEMENTWISE || !has_prod_v<Root>) {
      return false;
    } else if constexpr (Lift<Root, T, NIN>::count != 1) {
      return false;
    } else {
      using P = typename the_prod<Root>::type;
      return prod_of_leaves<P>::value &&
             others_plain<leaves_t<typename Lift<Root, T, NIN>::type>, NIN, T>();
    }
  }();
};

// Do two bound matrices of `es`-byte elements share memory (as whole spans)?
inline bool overlap(const Binding& x, const Binding& y, size_t es) {
  if (x.rows * x.cols == 0 || y.rows * y.cols == 0) return false;
  auto span = [es](const Binding& b) { return (size_t(b.ld) * size_t(b.cols - 1) + size_t(b.rows)) * es; };
  const uintptr_t p = reinterpret_cast<uintptr_t>(x.p), q = reinterpret_cast<uintptr_t>(y.p);
  return p < q + span(y) && q < p + span(x);
}

// Products from which copying unaligned 16-bit operands, and splitting FP32
// ones, pays (M N K; any size with blocks_per_sm given). With the library's
// GEMM and the pass after it on the other side: BF16 1001 x 301 x 1501 18.4
// against 18.3 us, 513 x 7001 x 513 22.8 against 37.3, 1501^3 25.1 against
// 55.4, 4001^3 148 against 848; FP32 257 x 3000 x 257 28.8 against 22.9,
// 1000 x 300 x 1500 33 against 39, 1500^3 61 against 119, 3000^3 250 against
// 858.
constexpr double kRelayoutMin = double(1 << 30), kSplitMin = double(1 << 28);
// FP32 products of fewer terms keep the library's GEMM (blocks_per_sm given:
// any): with few terms of one sign the planes' cuts and left-out products weigh
// more than FP32's roundings. Root mean square error in 2^-24 of the product at
// K = 16, 24, 32: 0.86, 0.85, 0.96 on the planes, 0.71, 0.75, 1.42 in FP32; K =
// 1: at most 2.3 and 1.0.
constexpr int64_t kSplitK = 32;

// Evaluates the whole tree with umma::k_gemm_umma. TMA wants 16-byte aligned
// bases and leading dimensions; an operand without them is first copied to a
// workspace that has (k_relayout16: 4 bytes moved per operand element, small
// beside a large product, where the library's kernels for such operands run at
// a fraction of the tensor cores' rate). So is, at any size, an operand that Z
// is written over: other tiles' loads of it may come after a tile's store.
// *used is false when the shapes disagree (the caller's library path reports
// it), for a bare or scaled product of unaligned operands (nothing to fuse), or
// without workspace.
template <class T, int NIN, class Root>
fx_status run_umma(fx_expr* x, const Root& root, cudaStream_t st, bool* used) {
  *used = false;
  using LR = Lift<Root, T, NIN>;
  using Lifted = typename LR::type;
  constexpr int PS = NIN;
  using P = typename the_prod<Root>::type;
  using OA = Operand<std::decay_t<decltype(std::declval<P>().l)>>;
  using OB = Operand<std::decay_t<decltype(std::declval<P>().r)>>;
  constexpr bool AMN = !OA::trans, BMN = OB::trans;
  const Binding& a = x->b[OA::slot];
  const Binding& b = x->b[OB::slot];
  const Binding& zb = x->b[NIN];
  if (!a.bound || !b.bound || !zb.bound) return FX_OK;
  const int64_t M = OA::trans ? a.cols : a.rows, Ka = OA::trans ? a.rows : a.cols;
  const int64_t Kb = OB::trans ? b.cols : b.rows, N = OB::trans ? b.rows : b.cols;
  if (Ka != Kb || zb.rows != M || zb.cols != N || M == 0 || N == 0 || Ka == 0) return FX_OK;
  const int64_t lim = int64_t(1) << 31;
  if (M >= lim || N >= lim || Ka >= lim ||
      ((M + umma::BM - 1) / umma::BM) * ((N + umma::BN - 1) / umma::BN) >= lim)
    return FX_OK;
  Binding bt[FX_MAX_SLOTS];
  for (int k = 0; k < NIN; ++k) bt[k] = x->b[k];
  bt[PS] = Binding{nullptr, M, N, M, true};
  if (check_leaves<leaves_t<Lifted>>(bt, M, N) != FX_OK) {
    cudaGetLastError();
    return FX_OK;  // the library-GEMM path reports the shape error
  }
  CUtensorMap ma, mb;
  const int sms = device_sms() > 0 ? device_sms() : 1;
  // Pairs of CTAs where their 256 x 256 tiles fill the chip in no more waves
  // than single CTAs' 128 x 256 ones do (8192^3 BF16: 683 us against 722)
  const int64_t ntiles = ((M + umma::BM - 1) / umma::BM) * ((N + umma::BN - 1) / umma::BN);
  const int64_t ptiles = ((M + umma::PBM - 1) / umma::PBM) * ((N + umma::BN - 1) / umma::BN);
  const bool pair = (ptiles * 2 + sms - 1) / sms <= (ntiles + sms - 1) / sms && ptiles * 2 >= sms;
  auto encode = [](CUtensorMap* m, const Binding& o, bool mn, int box) {
    return encode_map<T>(m, o.p, o.rows, o.cols, o.ld, 64, mn ? 64 : box);
  };
  const bool oka = encode(&ma, a, AMN, umma::BM), okb = encode(&mb, b, BMN, pair ? umma::BN / 2 : umma::BN);
  if ((!oka || !okb) &&
      (ScaledProd<Root>::value || (double(M) * double(N) * double(Ka) < kRelayoutMin && x->tune.bps == 0)))
    return FX_OK;
  const bool mova = !oka || overlap(zb, a, sizeof(T)), movb = !okb || overlap(zb, b, sizeof(T));
  umma::Relayout ca{}, cb{};
  if (mova || movb) {
    auto ldp = [](const Binding& o) { return (o.rows + 7) / 8 * 8; };
    auto bytes = [&](const Binding& o) { return (size_t(ldp(o)) * size_t(o.cols) * sizeof(T) + 255) & ~size_t(255); };
    auto copy = [&](const Binding& o, char* d) {
      const int64_t pc = (o.rows + 255) / 256;
      return umma::Relayout{o.p, d, o.rows, o.cols, o.ld, ldp(o), pc * o.cols, FastDiv::make(uint32_t(pc))};
    };
    const size_t na = mova ? bytes(a) : 0, nb = movb ? bytes(b) : 0;
    if (x->ws_gemm.ensure(na + nb, st) != FX_OK) {
      cudaGetLastError();
      return FX_OK;
    }
    char* w = static_cast<char*>(x->ws_gemm.p);
    auto moved = [&](const Binding& o, char* d) { return Binding{d, o.rows, o.cols, ldp(o), true}; };
    if (mova) {
      ca = copy(a, w);
      if (!encode(&ma, moved(a, w), AMN, umma::BM)) return FX_OK;
    }
    if (movb) {
      cb = copy(b, w + na);
      if (!encode(&mb, moved(b, w + na), BMN, pair ? umma::BN / 2 : umma::BN)) return FX_OK;
    }
    if (ca.items >= (int64_t(1) << 32) || cb.items >= (int64_t(1) << 32)) return FX_OK;
  }
  auto kern = umma::k_gemm_umma<T, AMN, BMN, Lifted, PS>;
  const int smem = umma::NS * umma::STAGE + 1024 + int(sizeof(umma::Bars));
  FX_TRY(allow_smem(kern, smem));
  FX_TRY(x->ws_err.ensure(256, st));
  unsigned int* err = static_cast<unsigned int*>(x->ws_err.p);
  const Slots sl = make_slots(x->b, NIN);
  const unsigned grid = unsigned(ntiles < sms ? ntiles : sms);   // persistent: one CTA per SM
  *used = true;
  x->last_launches = 0;
  if (ca.items + cb.items > 0) {
    const int64_t blocks = (ca.items + cb.items + 7) / 8;
    umma::k_relayout16<<<unsigned(blocks < sms * 8 ? blocks : sms * 8), 256, 0, st>>>(ca, cb);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "k_relayout16");
  }
  if (pair) {
    auto pk = umma::k_gemm_umma_pair<T, AMN, BMN, Lifted, PS>;
    const int psmem = umma::PNS * umma::PSTAGE + 1024 + int(sizeof(umma::PairBars));
    FX_TRY(allow_smem(pk, psmem));
    // as many pairs as can be resident: a tile processor may have an SM without a partner
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(sms / 2 * 2));
    cfg.blockDim = dim3(umma::THREADS);
    cfg.dynamicSmemBytes = size_t(psmem);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int pairs = 0;
    if (cudaOccupancyMaxActiveClusters(&pairs, pk, &cfg) != cudaSuccess || pairs < 1) {
      cudaGetLastError();
      pairs = 1;
    }
    if (pairs > sms / 2) pairs = sms / 2;
    if (pairs > ptiles) pairs = int(ptiles);
    pk<<<unsigned(2 * pairs), umma::THREADS, psmem, st>>>(ma, mb, LR::make(root), sl, static_cast<T*>(zb.p), zb.ld,
                                                int(M), int(N), int(Ka), err);
    const cudaError_t pe = cudaGetLastError();
    if (pe != cudaSuccess) return cuda_fail(pe, "k_gemm_umma_pair");
    x->last_launches = 1;
    return FX_OK;
  }
  kern<<<grid, umma::THREADS, smem, st>>>(ma, mb, LR::make(root), sl, static_cast<T*>(zb.p), zb.ld, int(M),
                                int(N), int(Ka), err);
  const cudaError_t le = cudaGetLastError();
  if (le != cudaSuccess) return cuda_fail(le, "k_gemm_umma");
  x->last_launches = 1;
  return FX_OK;
}

// FP32: the operands split into BF16 planes, then umma32::k_gemm_umma32 (two
// launches). Takes operands of any alignment and leading dimension, since
// the planes are laid out here. *used is false when the shapes disagree (the
// library path reports it), an extent is beyond the kernels' indices, or
// the workspace for the planes cannot be had (the library path needs less).
template <int NIN, class Root>
fx_status run_umma32(fx_expr* x, const Root& root, cudaStream_t st, bool* used) {
  namespace u3 = umma32;
  *used = false;
  using LR = Lift<Root, float, NIN>;
  using Lifted = typename LR::type;
  constexpr int PS = NIN;
  using P = typename the_prod<Root>::type;
  using OA = Operand<std::decay_t<decltype(std::declval<P>().l)>>;
  using OB = Operand<std::decay_t<decltype(std::declval<P>().r)>>;
  constexpr bool AMN = !OA::trans, BMN = OB::trans;
  const Binding& a = x->b[OA::slot];
  const Binding& b = x->b[OB::slot];
  const Binding& zb = x->b[NIN];
  if (!a.bound || !b.bound || !zb.bound) return FX_OK;
  const int64_t M = OA::trans ? a.cols : a.rows, K = OA::trans ? a.rows : a.cols;
  const int64_t Kb = OB::trans ? b.cols : b.rows, N = OB::trans ? b.rows : b.cols;
  if (K != Kb || zb.rows != M || zb.cols != N || M == 0 || N == 0 || K == 0) return FX_OK;
  const int64_t lim = int64_t(1) << 30;
  if (M >= lim || N >= lim || K >= lim) return FX_OK;
  if ((double(M) * double(N) * double(K) < kSplitMin || K < kSplitK) && x->tune.bps == 0) return FX_OK;
  // Z written over an operand: the fallback for unsplittable values reads the
  // operands while other blocks store
  if (overlap(zb, a, sizeof(float)) || overlap(zb, b, sizeof(float))) return FX_OK;
  const int sms = device_sms() > 0 ? device_sms() : 1;
  const u3::Shape32 shape = u3::choose_shape(M, N, int((K + u3::BK - 1) / u3::BK), sms);
  const int64_t ntiles = ((M + u3::BM - 1) / u3::BM) * ((N + shape.bn - 1) / shape.bn);
  const int64_t pieces = (int64_t(1) << 32) - 1;
  auto items = [](const Binding& o) { return (o.rows + 7) / 8 * o.cols; };
  if (ntiles >= (int64_t(1) << 26) || items(a) > pieces || items(b) > pieces) return FX_OK;
  Binding bt[FX_MAX_SLOTS];
  for (int k = 0; k < NIN; ++k) bt[k] = x->b[k];
  bt[PS] = Binding{nullptr, M, N, M, true};
  if (check_leaves<leaves_t<Lifted>>(bt, M, N) != FX_OK) {
    cudaGetLastError();
    return FX_OK;
  }
  const int S = shape.S;
  auto up = [](size_t v) { return (v + 255) & ~size_t(255); };
  auto ldp = [](const Binding& o) { return (o.rows + 7) / 8 * 8; };
  const size_t pa = up(size_t(ldp(a)) * size_t(a.cols) * 6), pb = up(size_t(ldp(b)) * size_t(b.cols) * 6);
  const size_t pp = S > 1 ? size_t(ntiles) * S * u3::BM * shape.bn * sizeof(float) : 0;
  if (x->ws_gemm.ensure(pa + pb + pp, st) != FX_OK) {
    cudaGetLastError();
    return FX_OK;
  }
  const Run r = run_of(x, st);
  unsigned int *tick = nullptr, *err = nullptr;
  // two words and the marks of the tile rows and columns (u3::Marks), then a ticket per tile
  const int64_t tiles_m = (M + u3::BM - 1) / u3::BM, nmarks = 2 + tiles_m + (N + shape.bn - 1) / shape.bn;
  FX_TRY(tickets(r, nmarks + ntiles, &tick));
  FX_TRY(err_word(r, &err));
  const u3::Marks marks{tick, tick + 2, tick + 2 + tiles_m};
  bf16* da = static_cast<bf16*>(x->ws_gemm.p);
  bf16* db = da + pa / 2;
  float* part = reinterpret_cast<float*>(db + pb / 2);
  u3::Maps maps;
  auto planes = [&](const Binding& o, bf16* d, int box1, std::initializer_list<int> at) {
    int64_t p = 0;
    for (int k : at)
      if (!encode_map<bf16>(&maps.m[k], d + p++ * ldp(o) * o.cols, o.rows, o.cols, ldp(o), 64, box1))
        return false;
    return true;
  };
  if (!planes(a, da, AMN ? 64 : u3::BM, {u3::A1, u3::A2, u3::A3}) ||
      !planes(b, db, BMN ? 64 : shape.bn, {u3::B1, u3::B2, u3::B3}))
    return FX_OK;
  auto split = [&](const Binding& o, bf16* d, unsigned int* m, bool mn, int tile) {
    return u3::SplitArgs{static_cast<const float*>(o.p), d, o.rows, o.cols, o.ld, ldp(o), items(o),
                         FastDiv::make(uint32_t((o.rows + 7) / 8)),
                         aligned(o.p, 16) && o.ld % 4 == 0 ? 1 : 0, m, mn ? 1 : 0, tile == 256 ? 8 : 7};
  };
  *used = true;
  x->last_launches = 0;
  const int64_t blocks = (items(a) + items(b) + 255) / 256;
  u3::k_split3<<<unsigned(blocks < sms * 8 ? blocks : sms * 8), 256, 0, st>>>(
      split(a, da, marks.rows, AMN, u3::BM), split(b, db, marks.cols, BMN, shape.bn), marks.any);
  // without the kernel that follows nothing clears the marks
  auto clear = [&](fx_status f) {
    if (f != FX_OK) cudaMemsetAsync(tick, 0, size_t(nmarks) * sizeof(unsigned int), st);
    return f;
  };
  FX_TRY(clear(after_launch(r, "k_split3")));
  x->last_launches = 0;  // counts launches that evaluate the tree, not those that lay out operands
  const int64_t nitems = ntiles * S;
  const u3::Source sa{static_cast<const float*>(a.p), AMN ? 1 : a.ld, AMN ? a.ld : 1};
  const u3::Source sb{static_cast<const float*>(b.p), BMN ? 1 : b.ld, BMN ? b.ld : 1};
  auto launch = [&](auto bn) -> fx_status {
    constexpr int BN = decltype(bn)::value;
    using SL = u3::Slots32<BN>;
    auto kern = u3::k_gemm_umma32<BN, AMN, BMN, Lifted, PS>;
    const int smem = int(SL::bytes) + 1024 + int(sizeof(u3::Bars));
    FX_TRY(allow_smem(kern, smem));
    kern<<<unsigned(nitems < sms ? nitems : sms), SL::THREADS, smem, st>>>(
        maps, LR::make(root), make_slots(x->b, NIN), static_cast<float*>(zb.p), zb.ld, int(M), int(N),
        int(K), S, part, tick + nmarks, marks, sa, sb, err);
    return after_launch(r, "k_gemm_umma32");
  };
  return clear(shape.bn == 256 ? launch(std::integral_constant<int, 256>{})
                               : launch(std::integral_constant<int, 128>{}));
}

// A tree with matrix products: products into temporaries (slots NIN ..
// NIN+P-1 of a private binding table), then the lifted tree on the fused
// path (or, for the unfused baseline, one launch per operator).
template <class T, int NIN, class Root>
fx_status run_with_prods(fx_expr* x, const Root& root, int kind, cudaStream_t st, bool unfused) {
  using LR = Lift<Root, T, NIN>;
  constexpr int P = LR::count;
  const int n_out = x->e->n_out;
  static_assert(NIN + P + 2 <= FX_MAX_SLOTS, "too many matrix products in one tree");
  using Inner = typename root_of<Root>::inner;
  const Inner& inner = inner_of(root);
  if constexpr (umma_ok<T, NIN, Root>::value) {
    // launch-shape pipeline 0: the tensor-core kernel with the remainder in
    // its epilogue; 1 and 2: the library GEMM and the fused pass
    if (!unfused && kind == FX_KIND_ELEMENTWISE && x->tune.pipe == 0) {
      bool used = false;
      if constexpr (!std::is_same<T, float>::value) {
        FX_TRY((run_umma<T, NIN>(x, root, st, &used)));
      } else if constexpr (!ScaledProd<Root>::value) {
        // a bare or scaled FP32 product has nothing to fuse: the library GEMM
        FX_TRY((run_umma32<NIN>(x, root, st, &used)));
      }
      if (used) return FX_OK;
    }
  }
  Binding bb[FX_MAX_SLOTS];
  for (int k = 0; k < NIN; ++k) bb[k] = x->b[k];
  for (int j = 0; j < n_out; ++j) bb[NIN + P + j] = x->b[NIN + j];
  size_t off = 0;
  if constexpr (ScaledProd<Root>::value) {
    using SP = ScaledProd<Root>;
    using PT = typename SP::P;
    using LA = Lift<decltype(PT::l), T, NIN>;
    using RA = Lift<decltype(PT::r), T, NIN + LA::count>;
    // straight into Z, unless Z lies over one of the last product's operands:
    // then by way of a temporary, as for other trees
    auto over = [&](int k) { return k < NIN && overlap(x->b[NIN], x->b[k], sizeof(T)); };
    const bool in_place = over(Operand<typename LA::type>::slot) || over(Operand<typename RA::type>::slot);
    if (!unfused && kind == FX_KIND_ELEMENTWISE && !in_place) {
      const PT& pr = SP::prod(root);
      FX_TRY((Prods<T, NIN, std::decay_t<decltype(pr.l)>>::run(bb, pr.l, nullptr, off, true, st)));
      FX_TRY((Prods<T, NIN + LA::count, std::decay_t<decltype(pr.r)>>::run(bb, pr.r, nullptr, off,
                                                                            true, st)));
      if (off > 0) FX_TRY(x->ws_gemm.ensure(off + 256, st));
      off = 0;
      char* base = static_cast<char*>(x->ws_gemm.p);
      FX_TRY((Prods<T, NIN, std::decay_t<decltype(pr.l)>>::run(bb, pr.l, base, off, false, st)));
      FX_TRY((Prods<T, NIN + LA::count, std::decay_t<decltype(pr.r)>>::run(bb, pr.r, base, off,
                                                                            false, st)));
      const Binding& z = x->b[NIN];
      x->last_launches = 0;
      return gemm_into<T, typename LA::type, typename RA::type>(bb, z.p, z.ld, z.rows, z.cols,
                                                                 SP::scale(root), st);
    }
  }
  FX_TRY((Prods<T, NIN, Inner>::run(bb, inner, nullptr, off, true, st)));
  if (off > 0) FX_TRY(x->ws_gemm.ensure(off + 256, st));
  off = 0;
  FX_TRY((Prods<T, NIN, Inner>::run(bb, inner, static_cast<char*>(x->ws_gemm.p), off, false, st)));
  Run r = run_of(x, st);
  r.b = bb;
  r.n_in = NIN + P;
  x->last_launches = 0;
  const auto lifted = LR::make(root);
  if (unfused) return run_unfused<T>(x, lifted, kind, st, &r);
  return run_root<T>(r, lifted, kind);
}

}  // namespace fx
