"""Performance cases of the library: what its users call, over the real range of sizes.

Every case is one pass through the public Python entry points of
`paper_1303_0270_gb300` (``ccm``, ``batch``) with the outputs and workspaces
allocated once, as a program that repeats the call keeps them.  Inputs are
drawn on the GPU from the seed alone.

listed()   the cases that are always measured
draw(rng)  one more case of the same ranges
prepare()  inputs, packed operands, outputs and workspaces of a case
run()      one pass; returns the result buffers (public header words + data words)
work()     bytes and operations a pass cannot do without
exact()    the same outputs from plain torch / numpy integer (or exact float64) arithmetic
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1303_0270_gb300 import ccm
from paper_1303_0270_gb300.batch import BatchMatvec

PUBLIC = 10  # header words a caller reads: magic, width, sign, status, rows, cols, nwords
M32 = 0xFFFFFFFF


def listed() -> list[dict]:
    return [
        # The smallest work: every operation once on 256 x 256 int32 matrices with
        # entries in [-100, 100] (the reference configuration of the tests).  Launches
        # and latency count.
        {"name": "small_chain_256", "op": "chain", "rows": 256, "cols": 256, "inner": 256},
        # Compressing a large count matrix (8192 x 8192, int64, Poisson(5)): the first
        # thing done with every matrix of the counting workload.
        {"name": "pack_8192_counts", "op": "pack", "rows": 8192, "cols": 8192,
         "dist": "counts", "width": 5, "bits": 64},
        # Compressing measurements that arrive as 32-bit integers, odd shape, wide fields.
        {"name": "pack_2999x5003_s21_i32", "op": "pack", "rows": 2999, "cols": 5003,
         "dist": "signed", "width": 21, "bits": 32},
        # Back to dense int64 from the middle of the width range.
        {"name": "unpack_8192_s12", "op": "unpack", "rows": 8192, "cols": 8192,
         "dist": "signed", "width": 12, "bits": 64},
        # Sum of two count matrices, result re-packed at its own width.
        {"name": "add_8192_counts", "op": "add", "rows": 8192, "cols": 8192,
         "dist": "counts", "width": 5, "width2": 5},
        # A matrix times a small factor, odd shape, signed fields.
        {"name": "scale_6007x7001_s9", "op": "scale", "rows": 6007, "cols": 7001,
         "dist": "signed", "width": 9, "factor": 7},
        # Matrix times vector on the count matrix: rows aligned to the kernels' chunks.
        {"name": "matvec_8192_counts", "op": "matvec", "rows": 8192, "cols": 8192,
         "dist": "counts", "width": 5, "widthx": 8},
        # Matrix times vector of the serving store, whose sizes are log-uniform: rows that
        # begin anywhere in a word.
        {"name": "matvec_20011x5003_s14", "op": "matvec", "rows": 20011, "cols": 5003,
         "dist": "signed", "width": 14, "widthx": 8},
        # The square matrix product of the matmul workload at 8 bits.
        {"name": "matmul_4096_s8", "op": "matmul", "rows": 4096, "cols": 4096, "inner": 4096,
         "dist": "signed", "width": 8, "width2": 8},
        # A matrix product of the serving store: odd sizes, widths at the top of its range
        # (2..20 bits).
        {"name": "matmul_3001x2503x3500_s20", "op": "matmul", "rows": 3001, "cols": 3500,
         "inner": 2503, "dist": "signed", "width": 20, "width2": 18},
        # 10,000 matrices of uneven shapes and widths, one product each, replayed as a
        # graph: the batched workload.
        {"name": "batch_10000", "op": "batch", "count": 10000, "shapes": 1303},
        # The variable-length encoding where it is the smaller one (bit lengths spread over
        # 1..40): encode, decode, and the product on the encoded form.
        {"name": "vlb_4096_tail40", "op": "vlb", "rows": 4096, "cols": 4096, "dist": "tail",
         "width": 40, "widthx": 8},
    ]


def draw(rng) -> dict:
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    rows, cols = logint(64, 8192), logint(64, 8192)
    dist = rng.choice(["signed", "unsigned", "counts"])
    width = 5 if dist == "counts" else rng.randint(1, 32)
    op = rng.choice(["chain", "pack", "unpack", "add", "scale", "matvec", "matvec", "matmul",
                     "matmul", "batch", "vlb"])
    if op == "chain":
        return {"op": op, "rows": logint(16, 512), "cols": logint(16, 512),
                "inner": logint(16, 512)}
    if op in ("pack", "unpack"):
        return {"op": op, "rows": rows, "cols": cols, "dist": dist, "width": width,
                "bits": rng.choice([32, 64]) if width < 32 else 64}
    if op == "add":
        w2 = width if dist == "counts" or rng.random() < 0.7 else rng.randint(1, 32)
        return {"op": op, "rows": rows, "cols": cols, "dist": dist, "width": width, "width2": w2}
    if op == "scale":
        return {"op": op, "rows": rows, "cols": cols, "dist": dist, "width": width,
                "factor": rng.choice([2, 3, 5, 7, -7, 12, 30, 100, -1000])}
    if op == "matvec":
        if rng.random() < 0.4:  # rows of whole 128-column chunks
            cols = max(128, cols // 128 * 128)
        return {"op": op, "rows": rows, "cols": cols, "dist": dist, "width": width,
                "widthx": rng.randint(4, 12)}
    if op == "matmul":
        while True:
            inner = logint(64, 8192)
            if rows * cols * inner <= 2503 * 3001 * 3500:
                break
            rows, cols = logint(64, 8192), logint(64, 8192)
        return {"op": op, "rows": rows, "cols": cols, "inner": inner,
                "dist": rng.choice(["signed", "unsigned"]), "width": rng.randint(2, 20),
                "width2": rng.randint(2, 20)}
    if op == "batch":
        return {"op": op, "count": logint(100, 10000), "shapes": rng.randint(1, 1 << 20)}
    return {"op": op, "rows": logint(64, 4096), "cols": logint(64, 4096), "dist": "tail",
            "width": rng.randint(8, 40), "widthx": 8}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _values(g, rows: int, cols: int, dist: str, width: int) -> torch.Tensor:
    if dist == "tail":  # bit lengths spread evenly over 1..width
        n = rows * cols
        top = torch.randperm(n, generator=g, device="cuda").remainder_(width)
        low = torch.randint(0, 1 << 62, (n,), generator=g, device="cuda", dtype=torch.int64)
        top = torch.ones_like(low) << top
        return (top + (low & (top - 1))).view(rows, cols)
    if dist == "counts":  # Poisson(5)
        lam = torch.full((rows, cols), 5.0, device="cuda")
        v = torch.poisson(lam, generator=g).to(torch.int64)
        lo, hi = 0, 20
    else:
        lo, hi = ((-(1 << (width - 1)), (1 << (width - 1)) - 1) if dist == "signed" else
                  (0, (1 << width) - 1))
        v = torch.randint(lo, hi + 1, (rows, cols), generator=g, device="cuda",
                          dtype=torch.int64)
    # the ends of the range, which a large matrix holds anyway: the width of the data (and
    # of sums and multiples) then does not hang on the seed
    v.view(-1)[0], v.view(-1)[-1] = hi, lo
    return v


def _generator(seed: int) -> torch.Generator:
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _dense(case: dict, seed: int) -> dict:
    """The dense int64 inputs of a case."""
    g, op = _generator(seed), case["op"]
    d = {}
    if op == "chain":
        m, n, k = case["rows"], case["cols"], case["inner"]
        for name, r, c in (("a", m, n), ("b", m, n), ("x", n, 1), ("c", n, k)):
            d[name] = torch.randint(-100, 101, (r, c), generator=g, device="cuda")
        d["idx"] = torch.randint(0, m * n, (1024,), generator=g, device="cuda")
        return d
    inner = case.get("inner")
    d["a"] = _values(g, case["rows"], inner or case["cols"], case["dist"], case["width"])
    if op == "add":
        d["b"] = _values(g, case["rows"], case["cols"], case["dist"], case["width2"])
    if op == "matmul":
        d["b"] = _values(g, inner, case["cols"], case["dist"], case["width2"])
    if op in ("matvec", "vlb"):
        d["x"] = _values(g, case["cols"], 1, "signed", case["widthx"])
    return d


def _product(a: torch.Tensor, b: torch.Tensor) -> torch.Tensor:
    """Integer product through float64: every partial sum is below 2^53, so exact."""
    return (a.double() @ b.double()).to(torch.int64)


def _results(case: dict, d: dict) -> dict:
    """The dense int64 results that a case packs."""
    op = case["op"]
    if op == "chain":
        return {"sum": d["a"] + d["b"], "scaled": 7 * d["a"], "y": _product(d["a"], d["x"]),
                "prod": _product(d["a"], d["c"])}
    if op == "pack":
        return {"out": d["a"]}
    if op == "add":
        return {"out": d["a"] + d["b"]}
    if op == "scale":
        return {"out": case["factor"] * d["a"]}
    if op in ("matvec", "vlb"):
        return {"out": _product(d["a"], d["x"])}
    if op == "matmul":
        return {"out": _product(d["a"], d["b"])}
    return {}


def _width(v: torch.Tensor) -> tuple[int, int]:
    """(width, is_signed) by the width rule."""
    lo, hi = int(v.min()), int(v.max())
    if lo < 0:
        return 1 + max(hi.bit_length() if hi > 0 else 0, (~lo).bit_length()), 1
    return max(1, hi.bit_length()), 0


def _nwords(v: torch.Tensor) -> int:
    return ccm.words_for(v.shape[0], v.shape[1], _width(v)[0])


class _Out:
    """A result buffer and the parts of it that hold the result: the header
    words a caller reads and the data words (`nwords` of them; all of the
    zeroed buffer where the result's width hangs on the seed)."""

    def __init__(self, rows: int, cols: int, capacity: int, nwords: int | None = None):
        self.m = ccm.PackedMatrix(rows, cols, capacity, "cuda")
        self.m.buf.zero_()
        end = ccm.HEADER_WORDS + (capacity if nwords is None else nwords)
        self.parts = [self.m.buf[:PUBLIC], self.m.buf[ccm.HEADER_WORDS:end]]


def _vector_arena(shapes, capacities):
    """Packed vectors side by side in one buffer."""
    sizes = [ccm.HEADER_WORDS + c for c in capacities]
    arena = torch.zeros(sum(sizes), dtype=torch.int32, device="cuda")
    out, at = [], 0
    for rows, cap, size in zip(shapes, capacities, sizes):
        m = ccm.PackedMatrix(rows, 1, 0, "cuda")
        m.capacity, m.buf = cap, arena[at:at + size]
        out.append(m)
        at += size
    return arena, out


# ---------------------------------------------------------------------------
# The batch: shapes log-uniform in [16, 2048), widths uniform in 1..24, x 8 bits
# ---------------------------------------------------------------------------
def _batch_shapes(case: dict):
    r = np.random.RandomState(case["shapes"])
    n = case["count"]
    dims = np.floor(16.0 * (2048.0 / 16.0) ** r.random_sample((n, 2))).astype(np.int64)
    return [(int(a), int(b), int(w)) for (a, b), w in zip(dims, r.randint(1, 25, n))]


def _batch_values(case: dict, seed: int):
    g = _generator(seed)
    for rows, cols, width in _batch_shapes(case):
        yield (rows, cols, width, _values(g, rows, cols, "signed", width),
               _values(g, cols, 1, "signed", 8))


def _y_width(cols: int, width: int) -> int:
    return int(ccm.lib().ccm_bound_matvec(width, 1, 8, 1, cols))


def _prepare_batch(case: dict, seed: int) -> dict:
    mats, xs, rows_of, caps = [], [], [], []
    for rows, cols, width, a, x in _batch_values(case, seed):
        for v, w, to in ((a, width, mats), (x, 8, xs)):
            m = ccm.PackedMatrix(v.shape[0], v.shape[1], ccm.words_for(*v.shape, w), "cuda")
            to.append(ccm.pack_into(v, m))
        rows_of.append(rows)
        caps.append(ccm.words_for(rows, 1, _y_width(cols, width)))
    arena, ys = _vector_arena(rows_of, caps)
    bm = BatchMatvec(mats, xs, ys)
    bm.autotune()
    bm.capture()
    return {"op": "batch", "bm": bm, "out": arena}


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------
def prepare(case: dict, seed: int) -> dict:
    op = case["op"]
    if op == "batch":
        return _prepare_batch(case, seed)
    d = _dense(case, seed)
    s = {"op": op}
    rows, cols = case["rows"], case["cols"]
    if op == "chain":
        for k in ("a", "b", "x", "c"):
            s["d" + k] = d[k].to(torch.int32)
            w = _width(d[k])[0]
            s[k] = _Out(*d[k].shape, ccm.words_for(*d[k].shape, w), _nwords(d[k]))
        for k in ("a", "b", "x", "c"):
            ccm.pack_into(s["d" + k], s[k].m)
        a, b, x, c = s["a"].m, s["b"].m, s["x"].m, s["c"].m
        k = case["inner"]
        s["sum"] = _Out(rows, cols, ccm.words_for(rows, cols, ccm.bound_add(a, b)),
                        _nwords(d["a"] + d["b"]))
        s["scaled"] = _Out(rows, cols, ccm.words_for(rows, cols, ccm.bound_scale(a, 7)),
                           _nwords(7 * d["a"]))
        s["y"] = _Out(rows, 1, ccm.words_for(rows, 1, ccm.bound_matvec(a, x)))
        s["prod"] = _Out(rows, k, ccm.words_for(rows, k, ccm.bound_matmul(a, c)))
        s["dense"] = torch.empty((rows, cols), dtype=torch.int64, device="cuda")
        s["idx"] = d["idx"]
        s["ws_mv"] = ccm.workspace(ccm.OP_MATVEC, rows, cols, 1, "cuda")
        s["ws_mm"] = ccm.workspace(ccm.OP_MATMUL, rows, cols, k, "cuda")
        return s
    if op == "pack":
        s["dense"] = d["a"].to(torch.int32 if case["bits"] == 32 else torch.int64)
        s["out"] = _Out(rows, cols, ccm.words_for(rows, cols, _width(d["a"])[0]),
                        _nwords(d["a"]))
        s["ws"] = ccm.workspace(ccm.OP_PACK, rows, cols, s["out"].m.capacity, "cuda")
        return s
    if op == "vlb":
        s["dense"] = d["a"]
        s["capacity"] = int(ccm.vlb_measure(d["a"]).nwords)
        s["x"] = ccm.pack(d["x"])
        s["y"] = _Out(rows, 1, ccm.words_for(rows, 1, 64))
        s["ws"] = ccm.workspace(ccm.OP_VLB_MATVEC, rows, cols, 0, "cuda")
        return s
    a = s["a"] = ccm.pack(d["a"])
    result = None
    if op == "unpack":
        s["dtype"] = torch.int32 if case["bits"] == 32 else torch.int64
        s["dense"] = torch.empty((rows, cols), dtype=s["dtype"], device="cuda")
        return s
    if op == "add":
        b = s["b"] = ccm.pack(d["b"])
        bound, result = ccm.bound_add(a, b), d["a"] + d["b"]
    elif op == "scale":
        s["factor"] = case["factor"]
        bound, result = ccm.bound_scale(a, s["factor"]), s["factor"] * d["a"]
    elif op == "matvec":
        x = s["x"] = ccm.pack(d["x"])
        bound, cols = ccm.bound_matvec(a, x), 1
        s["ws"] = ccm.workspace(ccm.OP_MATVEC, a.rows, a.cols, 1, "cuda")
    else:
        b = s["b"] = ccm.pack(d["b"])
        bound = ccm.bound_matmul(a, b)
        s["ws"] = ccm.workspace(ccm.OP_MATMUL, a.rows, a.cols, b.cols, "cuda")
    s["out"] = _Out(rows, cols, ccm.words_for(rows, cols, bound),
                    None if result is None else _nwords(result))
    return s


def run(s: dict):
    op = s["op"]
    if op == "chain":
        for k in ("a", "b", "x", "c"):
            ccm.pack_into(s["d" + k], s[k].m)
        a = s["a"].m
        dense = ccm.unpack(a, out=s["dense"], check=False)
        got = ccm.get(a, s["idx"], check=False)
        ccm.add_into(a, s["b"].m, s["sum"].m)
        ccm.scale_into(a, 7, s["scaled"].m)
        ccm.matvec_into(a, s["x"].m, s["y"].m, ws=s["ws_mv"])
        ccm.matmul_into(a, s["c"].m, s["prod"].m, ws=s["ws_mm"])
        return [s[k].parts for k in ("a", "b", "x", "c", "sum", "scaled", "y", "prod")] + [
            dense, got]
    if op == "pack":
        ccm.pack_into(s["dense"], s["out"].m, ws=s["ws"])
        return s["out"].parts
    if op == "unpack":
        return ccm.unpack(s["a"], dtype=s["dtype"], out=s["dense"], check=False)
    if op == "add":
        ccm.add_into(s["a"], s["b"], s["out"].m)
        return s["out"].parts
    if op == "scale":
        ccm.scale_into(s["a"], s["factor"], s["out"].m)
        return s["out"].parts
    if op == "matvec":
        ccm.matvec_into(s["a"], s["x"], s["out"].m, ws=s["ws"])
        return s["out"].parts
    if op == "matmul":
        ccm.matmul_into(s["a"], s["b"], s["out"].m, ws=s["ws"])
        return s["out"].parts
    if op == "batch":
        s["bm"].run()
        return s["out"]
    v = ccm.vlb_pack(s["dense"], capacity=s["capacity"])
    dense = ccm.vlb_unpack(v, check=False)
    ccm.vlb_matvec_into(v, s["x"], s["y"].m, ws=s["ws"])
    return [v.buf[:PUBLIC], v.buf[ccm.HEADER_WORDS:], v.index, dense, s["y"].parts]


# ---------------------------------------------------------------------------
# Work that no implementation can do without
# ---------------------------------------------------------------------------
def work(case: dict) -> dict:
    op = case["op"]
    if op == "batch":
        nbytes = flops = 0
        for rows, cols, width in _batch_shapes(case):
            by = width + 8 + cols.bit_length() // 2
            nbytes += (rows * cols * width + cols * 8 + rows * by) // 8
            flops += 2 * rows * cols
        return {"bytes": nbytes, "flops": flops}
    m, n = case["rows"], case["cols"]
    if op == "chain":
        k = case["inner"]
        # int32 in, 8-bit fields packed and read, the results of 9, 10, 22 and 22 bits
        nbytes = (4 * (2 * m * n + n + n * k) + 2 * m * n + n + n * k + 8 * m * n
                  + 1024 * 17 + (9 + 10) * m * n // 8 + 22 * (m + m * k) // 8)
        return {"bytes": nbytes, "flops": 2 * m * n * (k + 1)}
    b = case["width"]
    if op in ("pack", "unpack"):
        return {"bytes": m * n * (b + case["bits"]) // 8, "flops": 0}
    if op == "add":
        b2 = case["width2"]
        return {"bytes": m * n * (b + b2 + max(b, b2) + 1) // 8, "flops": 0}
    if op == "scale":
        return {"bytes": m * n * (2 * b + abs(case["factor"]).bit_length()) // 8, "flops": 0}
    if op == "matvec":
        by = b + case["widthx"] + n.bit_length() // 2
        return {"bytes": (m * n * b + n * case["widthx"] + m * by) // 8, "flops": 2 * m * n}
    if op == "matmul":
        k, b2 = case["inner"], case["width2"]
        bc = b + b2 + k.bit_length() // 2
        return {"bytes": (m * k * b + k * n * b2 + m * n * bc) // 8, "flops": 2 * m * n * k}
    # encode (dense in, stream out), decode (stream in, dense out), product (stream in);
    # a mean entry takes the prefix plus half the largest length
    bits = b.bit_length() + (b + 1) / 2
    return {"bytes": int(m * n * (16 + 3 * bits / 8)), "flops": 2 * m * n}


# ---------------------------------------------------------------------------
# The same outputs by plain arithmetic
# ---------------------------------------------------------------------------
def _header(magic: int, width: int, signed: int, rows: int, cols: int, nwords: int):
    w = [magic, width, signed, 0, rows & M32, rows >> 32, cols & M32, cols >> 32, nwords & M32,
         nwords >> 32]
    return np.array(w, dtype=np.uint32).view(np.int32)


def _pack_words(v: torch.Tensor, b: int) -> torch.Tensor:
    """Fields of b bits, least significant bit first, in 32-bit words padded to four."""
    n = v.numel()
    groups = (n + 31) // 32
    f = torch.zeros(groups * 32, dtype=torch.int64, device=v.device)
    f[:n] = v.reshape(-1)
    if b < 64:
        f &= (1 << b) - 1
    f = f.view(groups, 32)
    out = torch.zeros((groups, b + 2), dtype=torch.int64, device=v.device)
    for e in range(32):
        w, sh = divmod(e * b, 32)
        lo, hi = (f[:, e] & M32) << sh, ((f[:, e] >> 32) & M32) << sh
        out[:, w] |= lo & M32
        out[:, w + 1] |= ((lo >> 32) & M32) | (hi & M32)
        if w + 2 < b + 2:
            out[:, w + 2] |= (hi >> 32) & M32
    words = out[:, :b].reshape(-1)[:(n * b + 31) // 32]
    words = torch.nn.functional.pad(words, (0, -words.numel() % 4))
    return torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)


def _packed(v: torch.Tensor, bound: int | None = None) -> list:
    """Header and words of v; `bound`: the words padded with zeros to that width's count."""
    b, sgn = _width(v)
    words = _pack_words(v, b)
    header = _header(ccm.MAGIC, b, sgn, v.shape[0], v.shape[1], words.numel())
    if bound:
        words = torch.nn.functional.pad(words, (0, ccm.words_for(*v.shape, bound) - words.numel()))
    return [header, words]


def _product_bound(a: torch.Tensor, b: torch.Tensor) -> int:
    """The width a program allots to the product of a and b."""
    return int(ccm.lib().ccm_bound_matmul(*_width(a), *_width(b), a.shape[1]))


def _bit_length(v: torch.Tensor) -> torch.Tensor:
    """Bit length of non-negative int64 entries below 2^53; that of 0 is 1."""
    return torch.frexp(v.double())[1].to(torch.int64).clamp_(min=1)


def _exact_vlb(a: torch.Tensor) -> list:
    """Prefix (the bit length) then value, entry after entry; offsets of every 64th entry."""
    v = a.reshape(-1)
    n, length = v.numel(), _bit_length(v)
    k = int(length.max()).bit_length()
    size = length + k
    start = torch.cumsum(size, 0) - size
    total = int(start[-1] + size[-1])
    nwords = ((total + 31) // 32 + 3) & ~3
    words = torch.zeros(nwords + 3, dtype=torch.int64, device=v.device)
    bits = length | (v << k)  # at most 6 + 40 bits
    w, sh = start >> 5, start & 31
    lo, hi = (bits & M32) << sh, (bits >> 32) << sh
    # entries do not overlap, so adding their bits is OR-ing them
    words.index_add_(0, w, lo & M32)
    words.index_add_(0, w + 1, (lo >> 32) + (hi & M32))
    words.index_add_(0, w + 2, hi >> 32)
    words = words[:nwords]
    words = torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)
    index = torch.cat([start[::64], torch.tensor([total], device=v.device)])
    return [_header(ccm.VLB_MAGIC, k, 0, a.shape[0], a.shape[1], nwords), words, index, a]


def _exact_batch(case: dict, seed: int) -> torch.Tensor:
    rows_of, caps, ys = [], [], []
    for rows, cols, width, a, x in _batch_values(case, seed):
        rows_of.append(rows)
        caps.append(ccm.words_for(rows, 1, _y_width(cols, width)))
        # every vector on a group of 32 fields of its own, so it begins on a word
        ys.append(torch.nn.functional.pad(_product(a, x).view(-1), (0, -rows % 32)))
    ends = np.cumsum([len(y) for y in ys])
    flat = torch.cat(ys)
    folded, host = (flat ^ (flat >> 63)).cpu().numpy(), flat.cpu().numpy()
    packed, blocks = {}, []
    for rows, cap, end, y in zip(rows_of, caps, ends, ys):
        at = int(end) - len(y)
        orv, neg = int(np.bitwise_or.reduce(folded[at:end])), int(host[at:end].min() < 0)
        b = orv.bit_length() + 1 if neg else max(1, orv.bit_length())
        if b not in packed:
            packed[b] = _pack_words(flat, b).cpu().numpy()
        nwords = ccm.words_for(rows, 1, b)
        data = (rows * b + 31) // 32
        block = np.zeros(ccm.HEADER_WORDS + cap, dtype=np.int32)
        block[:PUBLIC] = _header(ccm.MAGIC, b, neg, rows, 1, nwords)
        block[PUBLIC:PUBLIC + 3] = np.array([orv & M32, orv >> 32, neg],
                                            dtype=np.uint32).view(np.int32)
        first = at // 32 * b
        block[ccm.HEADER_WORDS:ccm.HEADER_WORDS + data] = packed[b][first:first + data]
        blocks.append(block)
    return torch.from_numpy(np.concatenate(blocks))


def exact(case: dict, seed: int):
    op = case["op"]
    if op == "batch":
        return _exact_batch(case, seed)
    d = _dense(case, seed)
    r = _results(case, d)
    if op == "chain":
        return [_packed(d[k]) for k in ("a", "b", "x", "c")] + [
            _packed(r["sum"]), _packed(r["scaled"]),
            _packed(r["y"], _product_bound(d["a"], d["x"])),
            _packed(r["prod"], _product_bound(d["a"], d["c"])),
            d["a"], d["a"].reshape(-1)[d["idx"]]]
    if op == "unpack":
        return d["a"].to(torch.int32 if case["bits"] == 32 else torch.int64)
    if op == "vlb":
        return _exact_vlb(d["a"]) + [_packed(r["out"], 64)]
    if op in ("matvec", "matmul"):
        return _packed(r["out"], _product_bound(d["a"], d["x" if op == "matvec" else "b"]))
    return _packed(r["out"])
