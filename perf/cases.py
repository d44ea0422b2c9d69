"""The workloads whose speed is tracked, as calls of the public Python API.

Six families, each a piece of work a program has the library do:

  zs      Z = A%B + 3.5*exp(C) - trans(D) and s = accu(square(A-B)) in one pass
          (element-wise tree with a transposed operand, and a sum beside it);
  stats   Z = X%Y + sqrt(abs(W))/(1+exp(-V)), sum(X%Y, 0), max(abs(X-Y), 1) and
          norm(X-Y, 2) of the same matrices, one evaluation each;
  batch   Z = A%B + 0.5*trans(C) and s = accu(Z) over many matrices of uneven
          shapes, one batched call on the program's own stream;
  loss    a training step of L = accu(square(sigmoid(X%W + b) - Y)): the loss
          and its gradients with respect to X, W and b, on a handle that the
          program keeps;
  gemm    sigmoid(s*X*Y + W): a matrix product with an element-wise remainder;
  suite   element-wise expressions: four-way add, 2*(X.t()+Y) + 2*(X+Y.t()),
          0.75*A + (B+C).t() + log(D^2), swish and gelu.

Matrices are dense and column-major, of any row count.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2604_22242_gb300 as fx

STORAGE = {"f32": fx.FX_F32, "f64": fx.FX_F64, "bf16": fx.FX_BF16, "f16": fx.FX_F16}
TORCH = {"f32": torch.float32, "f64": torch.float64, "bf16": torch.bfloat16, "f16": torch.float16}
BYTES = {"f32": 4, "f64": 8, "bf16": 2, "f16": 2}
SUITE = (("add4", ("A1", "A2", "A3", "A4")), ("expr1", ("A1", "A2")),
         ("expr2", ("A1", "A2", "A3", "A4")), ("swish", ("A1",)), ("gelu", ("A1",)))


def listed():
    return [
        # one call on a block-sized matrix: launch and latency are all there is
        {"name": "zs_small_f32", "family": "zs", "dtype": "f32", "rows": 64, "cols": 48},
        # the everyday single-precision size: fits in L2, a few microseconds of work
        {"name": "zs_1024_f32", "family": "zs", "dtype": "f32", "rows": 1024, "cols": 1024},
        # the largest size in the half-width storage types
        {"name": "zs_16384_bf16", "family": "zs", "dtype": "bf16", "rows": 16384, "cols": 16384},
        # odd row and column counts in half precision: columns start at odd addresses
        {"name": "zs_odd_f16", "family": "zs", "dtype": "f16", "rows": 5003, "cols": 4999},
        # column, row and whole-matrix statistics beside the element-wise result
        {"name": "stats_8192_f32", "family": "stats", "dtype": "f32", "rows": 8192, "cols": 8192},
        # the same in double precision, with an odd row count
        {"name": "stats_odd_f64", "family": "stats", "dtype": "f64", "rows": 3001, "cols": 4096},
        # thousands of matrices of uneven shapes in one call
        {"name": "batch_4096_f32", "family": "batch", "dtype": "f32", "count": 4096, "hi": 2048},
        # a training step small enough for its fixed costs to show
        {"name": "loss_small_f32", "family": "loss", "dtype": "f32", "rows": 257, "cols": 129},
        # a training step in mixed precision at full size
        {"name": "loss_8192_bf16", "family": "loss", "dtype": "bf16", "rows": 8192, "cols": 8192},
        # a large product with its remainder on half-width operands
        {"name": "gemm_8192_bf16", "family": "gemm", "dtype": "bf16", "m": 8192, "n": 8192,
         "k": 8192},
        # a middle-sized product in single precision
        {"name": "gemm_mid_f32", "family": "gemm", "dtype": "f32", "m": 2048, "n": 1536,
         "k": 2048},
        # the single-precision expressions of the paper's comparison at its size
        {"name": "suite_10000_f32", "family": "suite", "dtype": "f32", "rows": 10000},
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(("zs", "stats", "batch", "loss", "gemm", "suite"))
    if family == "zs":
        return {"family": family, "dtype": rng.choice(("f32", "bf16", "f16")),
                "rows": _size(rng, 48, 12000), "cols": _size(rng, 48, 12000)}
    if family == "stats":
        return {"family": family, "dtype": rng.choice(("f32", "f64")),
                "rows": _size(rng, 64, 8192), "cols": _size(rng, 64, 8192)}
    if family == "batch":
        return {"family": family, "dtype": rng.choice(("f32", "bf16")),
                "count": _size(rng, 64, 4096), "hi": _size(rng, 128, 2048)}
    if family == "loss":
        return {"family": family, "dtype": rng.choice(("f32", "bf16")),
                "rows": _size(rng, 128, 8192), "cols": _size(rng, 128, 8192)}
    if family == "gemm":
        dtype = rng.choice(("bf16", "f16", "f32"))
        hi = 3072 if dtype == "f32" else 8192
        return {"family": family, "dtype": dtype, "m": _size(rng, 256, hi),
                "n": _size(rng, 256, hi), "k": _size(rng, 256, hi)}
    return {"family": family, "dtype": "f32", "rows": _size(rng, 256, 10000)}


# ---------------------------------------------------------------- inputs


def _matrix(gen, rows, cols, dtype, dist):
    """A column-major rows x cols matrix of one distribution, drawn on the GPU."""
    t = fx.colmajor(rows, cols, TORCH[dtype])
    flat = t.t().reshape(-1)  # a view of the same memory: rows are contiguous
    step = 1 << 26
    for at in range(0, flat.numel(), step):  # in pieces: the draws are in 32 or 64 bits
        part = flat[at:at + step]
        part.copy_(_values(gen, part.numel(), dist, torch.float64 if dtype == "f64" else torch.float32))
    return t


def _values(gen, n, dist, dt):
    if dist == "uniform":  # U[-1, 1]
        return torch.rand(n, generator=gen, device="cuda", dtype=dt).mul_(2).sub_(1)
    v = torch.randn(n, generator=gen, device="cuda", dtype=dt)
    if dist == "normal_half":
        return v.mul_(0.5)
    if dist in ("lognormal", "lognormal9"):  # lognormal(0, 1) of either sign; 9: capped at 9
        v = v.exp_()
        if dist == "lognormal9":
            v = v.clamp_(max=9.0)
        sign = torch.rand(n, generator=gen, device="cuda") < 0.5
        return torch.where(sign, -v, v)
    return v


def _shapes(case):
    """Rows and columns of a batch, each log-uniform in [16, hi]."""
    rng = np.random.default_rng(1234 + case["count"])  # the shapes belong to the case
    rc = np.rint(np.exp(rng.uniform(math.log(16), math.log(case["hi"]), (case["count"], 2))))
    return rc.astype(np.int64)


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    f, d = case["family"], case["dtype"]
    if f == "zs":
        r, c = case["rows"], case["cols"]
        wide = d in ("bf16", "f16")
        dist = "lognormal" if wide else "uniform"
        # 3.5*exp(9) is finite in every storage type
        return {"A": _matrix(gen, r, c, d, dist), "B": _matrix(gen, r, c, d, dist),
                "C": _matrix(gen, r, c, d, "lognormal9" if wide else dist),
                "D": _matrix(gen, c, r, d, dist)}
    if f == "stats":
        return {k: _matrix(gen, case["rows"], case["cols"], d, "normal") for k in "XYWV"}
    if f == "loss":
        r, c = case["rows"], case["cols"]
        ins = {k: _matrix(gen, r, c, d, "normal_half") for k in "XWY"}
        ins["b"] = _matrix(gen, r, 1, d, "normal_half").reshape(-1)
        return ins
    if f == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"X": _matrix(gen, m, k, d, "normal"), "Y": _matrix(gen, k, n, d, "normal"),
                "W": _matrix(gen, m, n, d, "normal")}
    if f == "suite":
        n = case["rows"]
        return {f"A{k}": _matrix(gen, n, n, d, "uniform") for k in range(1, 5)}
    rc = _shapes(case)  # batch: every operand in one arena, matrices 16-byte aligned
    w = 16 // BYTES[d]
    sizes = (rc[:, 0] * rc[:, 1] + w - 1) // w * w
    offs = sizes.cumsum() - sizes
    ins = {k: _matrix(gen, int(sizes.sum()), 1, d, "uniform").reshape(-1) for k in "ABC"}
    ins["rc"], ins["offs"], ins["total"] = rc, offs, int(sizes.sum())
    return ins


class _State:
    pass


def _expr(name, dtype, ins, outs):
    ex = fx.Expr(name, STORAGE[dtype])
    for k, t in enumerate(ins):
        ex.bind(k, t)
    for k, t in enumerate(outs):
        ex.bind(ex.n_in + k, t)
    return ex


def prepare(case, seed):
    s = _State()
    s.case = case
    f, d = case["family"], case["dtype"]
    ins = s.ins = _inputs(case, seed)
    rdt = torch.float64 if d == "f64" else torch.float32
    if f == "zs":
        z, acc = fx.colmajor(case["rows"], case["cols"], TORCH[d]), fx.colmajor(1, 1, rdt)
        s.ex = _expr("schur_exp_trans_sqdiff", d, [ins[k] for k in "ABCD"], [z, acc])
        s.out = {"Z": z, "s": acc}
    elif f == "stats":
        r, c = case["rows"], case["cols"]
        s.out = {"Z": fx.colmajor(r, c, TORCH[d]), "colsum": fx.colmajor(1, c, rdt),
                 "rowmax": fx.colmajor(r, 1, rdt), "nrm": fx.colmajor(1, 1, rdt)}
        s.ex = [_expr(name, d, [ins[k] for k in slots], [s.out[out]])
                for name, slots, out in (("schur_sqrt_sigmoid", "XYWV", "Z"),
                                         ("schur_colsum", "XY", "colsum"),
                                         ("absdiff_rowmax", "XY", "rowmax"),
                                         ("diff_norm", "XY", "nrm"))]
    elif f == "batch":
        n, es = case["count"], BYTES[d]
        s.out = {"Z": torch.zeros(ins["total"], dtype=TORCH[d], device="cuda"),
                 "s": torch.zeros(n, dtype=rdt, device="cuda")}
        s.h = fx.Expr("schur_trans_accu", STORAGE[d])
        s.items = (fx.BatchItem * n)()
        base = [t.data_ptr() for t in (ins["A"], ins["B"], ins["C"], s.out["Z"])]
        for i, ((r, c), o) in enumerate(zip(ins["rc"].tolist(), ins["offs"].tolist())):
            it = s.items[i]
            for k in range(4):
                it.ptr[k] = base[k] + o * es
            it.ptr[4] = s.out["s"].data_ptr() + i * s.out["s"].element_size()
            it.rows, it.cols = r, c
        s.stream = torch.cuda.Stream()
        s.stream.wait_stream(torch.cuda.current_stream())
    elif f == "loss":
        r, c = case["rows"], case["cols"]
        s.out = {"L": fx.colmajor(1, 1, rdt), "gX": fx.colmajor(r, c, TORCH[d]),
                 "gW": fx.colmajor(r, c, TORCH[d]),
                 "gb": torch.empty(r, dtype=TORCH[d], device="cuda")}
        s.ex = _expr("sigmoid_sqloss", d, [ins[k] for k in "XWYb"], [s.out["L"]])
        # one gradient per input slot; Y is data and gets none
        s.grads = [s.out["gX"].data_ptr(), s.out["gW"].data_ptr(), 0, s.out["gb"].data_ptr()]
    elif f == "gemm":
        z = fx.colmajor(case["m"], case["n"], TORCH[d])
        s.ex = _expr("gemm_epilogue", d, [ins[k] for k in "XYW"], [z])
        s.ex.set_scalar(0, 1.0 / math.sqrt(case["k"]))
        s.out = {"Z": z}
    else:
        n = case["rows"]
        s.out = {name: fx.colmajor(n, n, TORCH[d]) for name, _ in SUITE}
        s.ex = [_expr(name, d, [ins[k] for k in slots], [s.out[name]]) for name, slots in SUITE]
    return s


def run(s):
    f = s.case["family"]
    if f in ("zs", "gemm"):
        s.ex.eval()
        return s.out
    if f in ("stats", "suite"):
        for ex in s.ex:
            ex.eval()
        return s.out
    if f == "batch":
        fx.fx_eval_batch(s.h.h, s.items, int(s.stream.cuda_stream), True)
        return s.out
    s.ex.eval()
    fx.fx_eval_backward(s.ex.h, 0, s.grads, int(torch.cuda.current_stream().cuda_stream))
    return s.out


def work(case):
    f, es = case["family"], BYTES[case["dtype"]]
    rb = 8 if case["dtype"] == "f64" else 4
    if f == "zs":
        n = case["rows"] * case["cols"]
        return {"bytes": 5 * n * es + rb, "flops": 8 * n}
    if f == "stats":
        # each of the four calls reads its own inputs
        n = case["rows"] * case["cols"]
        return {"bytes": 11 * n * es + (case["rows"] + case["cols"] + 1) * rb, "flops": 16 * n}
    if f == "batch":
        rc = _shapes(case)
        n = int((rc[:, 0] * rc[:, 1]).sum())
        return {"bytes": 4 * n * es + case["count"] * rb, "flops": 4 * n}
    if f == "loss":
        # forward reads X, W, Y; backward reads them again and writes gX, gW
        n = case["rows"] * case["cols"]
        return {"bytes": 8 * n * es + 3 * case["rows"] * es + rb, "flops": 24 * n}
    if f == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": (m * k + k * n + 2 * m * n) * es, "flops": 2 * m * n * k + 6 * m * n}
    n = case["rows"] ** 2
    return {"bytes": (5 + 3 + 5 + 2 + 2) * n * es, "flops": 40 * n}


def exact(case, seed):
    """The same results in 64 bits, by plain torch."""
    f = case["family"]
    ins = _inputs(case, seed)
    if f == "batch":
        z = torch.zeros(ins["total"], dtype=torch.float64, device="cuda")
        acc = []
        for (r, c), o in zip(ins["rc"].tolist(), ins["offs"].tolist()):
            a, b, t = (ins[k][o:o + r * c].double() for k in "ABC")
            v = a * b + 0.5 * t.view(r, c).t().reshape(-1)
            z[o:o + r * c] = v
            acc.append(v.sum())
        return {"Z": z, "s": torch.stack(acc)}
    v = {k: t.double() for k, t in ins.items()}
    if f == "zs":
        return {"Z": v["A"] * v["B"] + 3.5 * v["C"].exp() - v["D"].t(),
                "s": (v["A"] - v["B"]).square().sum().reshape(1, 1)}
    if f == "stats":
        xy, df = v["X"] * v["Y"], v["X"] - v["Y"]
        return {"Z": xy + v["W"].abs().sqrt() / (1 + (-v["V"]).exp()),
                "colsum": xy.sum(0, keepdim=True), "rowmax": df.abs().amax(1, keepdim=True),
                "nrm": df.square().sum().sqrt().reshape(1, 1)}
    if f == "loss":
        p = torch.sigmoid(v["X"] * v["W"] + v["b"][:, None])
        d = p - v["Y"]
        g = 2 * d * p * (1 - p)
        return {"L": d.square().sum().reshape(1, 1), "gX": g * v["W"], "gW": g * v["X"], "gb": g.sum(1)}
    if f == "gemm":
        return {"Z": torch.sigmoid(v["X"] @ v["Y"] / math.sqrt(case["k"]) + v["W"])}
    a1, a2, a3, a4 = (v[f"A{k}"] for k in range(1, 5))
    return {"add4": a1 + a2 + a3 + a4, "expr1": 2 * (a1.t() + a2) + 2 * (a1 + a2.t()),
            "expr2": 0.75 * a1 + (a2 + a3).t() + a4.square().log(),
            "swish": a1 * torch.sigmoid(a1),
            "gelu": a1 / 2 * (1 + torch.tanh(math.sqrt(2 / math.pi) * (a1 + 0.044715 * a1 ** 3)))}
