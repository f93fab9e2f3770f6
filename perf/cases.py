"""The work that users of the library have it do, as cases to be timed.

Each case is one pass through the public binding
(`paper_1410_6685_gb300.safegpu`): the paper's vector addition with its
postcondition, filter, sort, matrix product, Gaussian elimination, and the
batched collections, over sizes from the paper's smallest (10^3 elements) to
the largest of this repository's benchmark.  Contracts are on, as they are by
default: every product, sort and solve carries its built-in postcondition.

A pass returns what a program would go on with: views of the library's own
result buffers (no copy), each releasing its handle when the last view of it
is dropped, and the scalars it reads.
"""
from __future__ import annotations

import math

import torch

from paper_1410_6685_gb300 import inputs
from paper_1410_6685_gb300 import safegpu as sg

_PREC = {"f32": sg.SG_PREC_F32_SIMT, "bf16": sg.SG_PREC_BF16_TC, "f16": sg.SG_PREC_F16_TC}

# a program's expressions: z = x + y, its postcondition z == x + y, the
# filter's predicate, and the batched chain's map, precondition and filter
_ADD = [("x", 0), ("x", 1), ("add",)]
_ADD_POST = [("x", 0), ("x", 1), ("x", 2), ("add",), ("eq",)]
_CHAIN = ([("x", 0), ("x", 0), ("c", 1.0), ("fma",)], [("x", 0), ("c", 1.0), ("ge",)],
          [("x", 0), ("c", 1.5), ("gt",)])


def listed():
    return [
        # the paper's smallest vectors: nothing but calls, launches and latency
        {"name": "vadd_1e3", "kind": "vadd", "n": 1000},
        # the benchmark's streaming size: add, check every element, sum
        {"name": "vadd_2e28", "kind": "vadd", "n": 1 << 28},
        # the benchmark's filter: x > 0.25 keeps 37.5% of the items
        {"name": "filter_2e28", "kind": "filter", "n": 1 << 28, "above": 0.25},
        # the headline sort, with sortedness and permutation checked
        {"name": "sort_i32_2e26", "kind": "sort", "n": 1 << 26, "dtype": "i32", "distinct": 0},
        # the paper's quicksort type (REAL_32) at an ordinary, odd size
        {"name": "sort_f32_1e6", "kind": "sort", "n": 1000003, "dtype": "f32", "distinct": 0},
        # the paper's largest product (10^6 elements) in the default precision
        {"name": "matmul_f32_1000", "kind": "matmul", "m": 1000, "n": 1000, "k": 1000,
         "prec": "f32"},
        # a large product in the default precision
        {"name": "matmul_f32_4096", "kind": "matmul", "m": 4096, "n": 4096, "k": 4096,
         "prec": "f32"},
        # the benchmark's largest product, bf16 operands, Freivalds check
        {"name": "matmul_bf16_8192", "kind": "matmul", "m": 8192, "n": 8192, "k": 8192,
         "prec": "bf16"},
        # a ragged rectangular product (no built-in check: not square)
        {"name": "matmul_f16_ragged", "kind": "matmul", "m": 1537, "n": 1023, "k": 2049,
         "prec": "f16"},
        # the paper's largest elimination: a general matrix, interchanges in
        # every column, binary32 updates
        {"name": "solve_f32_1000", "kind": "solve", "n": 1000, "prec": "f32", "dominant": False},
        # the benchmark's largest elimination: diagonally dominant, bf16 updates
        {"name": "solve_bf16_8192", "kind": "solve", "n": 8192, "prec": "bf16", "dominant": True},
        # ten thousand collections of uneven size in one launch
        {"name": "batch_10000", "kind": "batch", "nseg": 10000},
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi], odd or even alike."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["vadd", "filter", "sort", "matmul", "matmul", "solve", "batch"])
    if kind == "vadd":
        return {"kind": kind, "n": _log_int(rng, 1000, 1 << 28)}
    if kind == "filter":
        return {"kind": kind, "n": _log_int(rng, 1000, 1 << 28),
                "above": round(rng.uniform(-0.9, 0.9), 3)}
    if kind == "sort":
        return {"kind": kind, "n": _log_int(rng, 1000, 1 << 26),
                "dtype": rng.choice(["i32", "f32"]), "distinct": rng.choice([0, 0, 256])}
    if kind == "matmul":
        prec = rng.choice(["f32", "bf16", "f16"])
        top = 4096 if prec == "f32" else 8192
        if rng.random() < 0.5:
            n = _log_int(rng, 200, top)
            return {"kind": kind, "m": n, "n": n, "k": n, "prec": prec}
        return {"kind": kind, "m": _log_int(rng, 200, top), "n": _log_int(rng, 200, top),
                "k": _log_int(rng, 64, top), "prec": prec}
    if kind == "solve":
        if rng.random() < 0.5:
            return {"kind": kind, "n": _log_int(rng, 100, 3000), "prec": "f32", "dominant": False}
        return {"kind": kind, "n": _log_int(rng, 100, 8192),
                "prec": rng.choice(["f32", "bf16", "f16"]) if rng.random() < 0.5 else "bf16",
                "dominant": True}
    return {"kind": kind, "nseg": _log_int(rng, 1000, 10000)}


# ---- what a program holds ----------------------------------------------------
_ctx = None


def _context():
    """The program's one context, on torch's current stream."""
    global _ctx
    if _ctx is None:
        _ctx = sg.sg_init(torch.cuda.current_device(), torch.cuda.current_stream().cuda_stream)
    return _ctx


class _Result:
    """A result handle of the library, for torch to view: torch keeps this
    object as long as the view lives, and the handle goes with it."""

    def __init__(self, release, handle, ptr, shape, typestr):
        self._release, self._handle = release, handle
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": tuple(shape),
                                         "typestr": typestr, "version": 3}

    def __del__(self):
        self._release(self._handle)


def _view(ctx, handle, shape, dtype):
    """A torch view of a result's own buffer (no copy), owning its handle."""
    matrix = len(shape) == 2
    release = sg.sg_matrix_release if matrix else sg.sg_vector_release
    if 0 in shape:
        release(handle)
        return torch.empty(shape, dtype=dtype, device="cuda")
    ptr = (sg.sg_matrix_device_ptr if matrix else sg.sg_vector_device_ptr)(ctx, handle)
    ts = {torch.float32: "<f4", torch.float64: "<f8", torch.int32: "<i4"}[dtype]
    return torch.as_tensor(_Result(release, handle, ptr, shape, ts), device="cuda")


class State:
    """Inputs on the device and the handles that wrap them."""

    def __init__(self, case):
        self.case = case
        self.ctx = _context()
        self.tensors = []
        self.handles = []

    def wrap(self, t):
        self.tensors.append(t)
        h = sg.wrap_tensor(self.ctx, t)
        self.handles.append((sg.sg_matrix_release if t.dim() == 2 else sg.sg_vector_release, h))
        return h

    def __del__(self):
        for release, h in self.handles:
            release(h)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(n, g):
    return torch.rand(n, device="cuda", generator=g).mul_(2.0).sub_(1.0)


def _shuffled_uniform(n, g):
    """n equidistant values of (-1, 1) in random order: a filter keeps the
    same number of them whatever the order."""
    p = torch.randperm(n, device="cuda", generator=g).double()
    return p.add_(0.5).mul_(2.0 / n).sub_(1.0).float()


def _keys(case, seed):
    """int32 keys over the whole range, or binary32 N(0, 1) keys; with
    `distinct`, drawn from that many values."""
    g, n = _gen(seed), case["n"]
    m = case["distinct"] or n
    if case["dtype"] == "i32":
        v = torch.randint(-2**31, 2**31, (m,), device="cuda", generator=g, dtype=torch.int32)
    else:
        v = torch.randn(m, device="cuda", generator=g)
    if case["distinct"]:
        v = v[torch.randint(0, m, (n,), device="cuda", generator=g)]
    return v.contiguous()


def _operands(case, seed):
    g = _gen(seed)
    return (torch.randn(case["m"], case["k"], device="cuda", generator=g),
            torch.randn(case["k"], case["n"], device="cuda", generator=g))


def _system(case, seed):
    """A x = b: off-diagonal N(0, 1); dominant: the diagonal is the row's
    absolute sum plus one and x is all ones; else x ~ N(0, 1)."""
    g, n = _gen(seed), case["n"]
    A = torch.randn(n, n, device="cuda", generator=g)
    if case["dominant"]:
        A.fill_diagonal_(0.0)
        A.diagonal().copy_(A.double().abs().sum(dim=1) + 1.0)
        return A, A.double().sum(dim=1)
    x = torch.randn(n, device="cuda", generator=g, dtype=torch.float64)
    return A, A.double() @ x


def _segments(case, seed):
    """Collections with lengths log-uniform in [2^6, 2^20], x ~ U[-1, 1)."""
    off = inputs.batch_offsets(inputs.batch_lengths(case["nseg"], seed))
    return _uniform(int(off[-1]), _gen(seed)), torch.from_numpy(off).cuda()


def prepare(case, seed):
    s = State(case)
    kind = case["kind"]
    if kind == "vadd":
        g = _gen(seed)
        s.x, s.y = s.wrap(_uniform(case["n"], g)), s.wrap(_uniform(case["n"], g))
        s.post = sg.contract(sg.SG_C_FOR_ALL, _ADD_POST, other=[s.x, s.y])
    elif kind == "filter":
        s.x = s.wrap(_shuffled_uniform(case["n"], _gen(seed)))
        s.pred = sg.expr([("x", 0), ("c", case["above"]), ("gt",)])
    elif kind == "sort":
        s.x = s.wrap(_keys(case, seed))
    elif kind == "matmul":
        a, b = _operands(case, seed)
        s.a, s.b = s.wrap(a), s.wrap(b)
    elif kind == "solve":
        A, b = _system(case, seed)
        s.a, s.b = s.wrap(A), s.wrap(b)
        s.opts = sg.SgSolveOpts()
        s.opts.precision = _PREC[case["prec"]]
    else:
        s.data, s.offsets = _segments(case, seed)
        n = case["nseg"]
        s.sums = torch.empty(n, dtype=torch.float64, device="cuda")
        s.first = torch.empty(n, dtype=torch.int64, device="cuda")
        s.kept = torch.empty(n, dtype=torch.int64, device="cuda")
        s.chain = sg.chain(*_CHAIN)
    return s


def run(s):
    case, ctx = s.case, s.ctx
    kind = case["kind"]
    if kind == "vadd":
        z = sg.sg_zip(ctx, _ADD, s.x, s.y)
        sg.sg_ensure(ctx, z, s.post)
        total = sg.sg_reduce(ctx, sg.SG_REDUCE_SUM, z)
        value = sg.sg_scalar_get(ctx, total)
        sg.sg_scalar_release(total)
        return {"z": _view(ctx, z, (case["n"],), torch.float32), "sum": value}
    if kind == "filter":
        k = sg.sg_filter(ctx, s.pred, s.x)
        return _view(ctx, k, (sg.sg_vector_count(ctx, k),), torch.float32)
    if kind == "sort":
        o = sg.sg_sort(ctx, s.x)
        return _view(ctx, o, (case["n"],), torch.int32 if case["dtype"] == "i32" else torch.float32)
    if kind == "matmul":
        c = sg.sg_matmul(ctx, s.a, s.b, _PREC[case["prec"]])
        return _view(ctx, c, (case["m"], case["n"]), torch.float32)
    if kind == "solve":
        x, _ = sg.sg_solve(ctx, s.a, s.b, s.opts)
        return _view(ctx, x, (case["n"],), torch.float64)
    sg.sg_batch_run(ctx, s.chain, s.data.data_ptr(), s.offsets.data_ptr(), case["nseg"],
                    s.sums.data_ptr(), s.first.data_ptr(), s.kept.data_ptr())
    return {"sums": s.sums, "first": s.first, "kept": s.kept}


def work(case):
    kind = case["kind"]
    if kind == "vadd":
        return {"bytes": 12 * case["n"], "flops": 2 * case["n"]}
    if kind == "filter":   # the kept share of the items is written
        return {"bytes": int(4 * case["n"] * (1 + (1 - case["above"]) / 2)), "flops": case["n"]}
    if kind == "sort":
        return {"bytes": 8 * case["n"], "flops": 0}
    if kind == "matmul":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 4 * (m * k + k * n + m * n), "flops": 2 * m * n * k}
    if kind == "solve":
        n = case["n"]
        return {"bytes": 4 * n * n + 16 * n, "flops": 2 * n**3 // 3}
    # the mean of 2^(6 + 14 u), u ~ U[0, 1)
    total = int(case["nseg"] * (2**20 - 2**6) / (14 * math.log(2)))
    return {"bytes": 4 * total + 24 * case["nseg"], "flops": 3 * total}


def exact(case, seed):
    kind = case["kind"]
    if kind == "vadd":
        g = _gen(seed)
        x, y = _uniform(case["n"], g), _uniform(case["n"], g)
        # the sum is of the binary32 z, as the pass computes it
        return {"z": x.double() + y.double(), "sum": float((x + y).double().sum())}
    if kind == "filter":
        x = _shuffled_uniform(case["n"], _gen(seed))
        return x[x > torch.tensor(case["above"], dtype=torch.float32, device="cuda")].double()
    if kind == "sort":
        v = torch.sort(_keys(case, seed)).values
        return v if case["dtype"] == "i32" else v.double()
    if kind == "matmul":
        a, b = _operands(case, seed)
        dt = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[case["prec"]]
        # operands rounded as the chosen precision states, the product in 64 bits
        return a.to(dt).double() @ b.to(dt).double()
    if kind == "solve":
        A, b = _system(case, seed)
        return torch.linalg.solve(A.double(), b)
    x, off = _segments(case, seed)
    y = torch.addcmul(torch.ones((), dtype=torch.float64, device="cuda"), x.double(), x.double())
    y = y.float()
    y = torch.where(y > 1.5, y, torch.zeros_like(y)).double()
    sums = torch.segment_reduce(y, "sum", lengths=off[1:] - off[:-1], unsafe=True)
    return {"sums": sums, "first": None, "kept": None}
