"""x of more than 14 bits (no byte image) on rows of a few and of many segments:
one matrix and batches of them, every width that a field can have, both signs, at
the edges of segments and stages, against the oracle word for word (integer work:
tolerance 0)."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import assert_same_packed, device, lib_ccm, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ccm():
    device()
    return lib_ccm()


def _rand(seed, shape, b, signed):
    lo, hi = synth.signed_range(b) if signed else (0, (1 << b) - 1)
    v = synth.uniform_int(seed, 0, int(np.prod(shape)), lo, hi).reshape(shape)
    v.flat[0], v.flat[-1] = hi, lo  # the width is b exactly
    return v


def _pack(ccm, v, b):
    m = ccm.PackedMatrix(v.shape[0], v.shape[1], ccm.words_for(*v.shape, b), device())
    return ccm.pack_into(to_dev(v), m)


# (rows, columns): 1 to 16 segments a row, whole and ragged, more rows than a stage holds
SHAPES = [(300, 1), (300, 2), (300, 3), (700, 16), (257, 31), (64, 32), (300, 33), (100, 64),
          (90, 97), (41, 200), (33, 224), (50, 225), (37, 256), (20, 257), (40, 480), (19, 481)]
X = [(15, 1), (15, 0), (24, 1), (31, 0), (8, 1)]  # (8 bits: int32 too at 16 and 32 bits of A)


def _oracle(a, x):
    try:
        return oracle.matvec(oracle.pack(a), oracle.pack(x))
    except OverflowError:  # (the widest pairs pass int64)
        return None


@pytest.mark.parametrize("b", list(range(1, 33)))
@pytest.mark.parametrize("sa", [0, 1])
def test_batch(ccm, b, sa):
    from paper_1303_0270_gb300.batch import BatchMatvec
    mats, xs, want = [], [], []
    for i, (m, n) in enumerate(SHAPES):
        for bx, sx in X:
            if b + bx + n.bit_length() > 63:
                continue  # (refused by the batch)
            mats.append(_rand(100 * b + i, (m, n), b, sa))
            xs.append(_rand(7 * bx + i, (n, 1), bx, sx))
            want.append(_oracle(mats[-1], xs[-1]))
    for unit, slots, stage in ((256, 0, 0), (32, 2, 128), (1024, 4, 1536)):
        ys = [ccm.PackedMatrix(a.shape[0], 1, ccm.words_for(a.shape[0], 1, 64), device())
              for a in mats]
        bm = BatchMatvec([_pack(ccm, a, b) for a in mats],
                         [ccm.pack(to_dev(x)) for x in xs], ys, unit_segments=unit)
        bm.slots, bm.stage_bytes = slots, stage
        bm.launch()
        torch.cuda.synchronize()
        for y, a, x, o in zip(ys, mats, xs, want):
            assert_same_packed(y, o, f"{a.shape} {b}/{sa}, unit {unit}")


@pytest.mark.parametrize("b,sa", [(1, 0), (2, 1), (5, 0), (13, 1), (16, 1), (17, 0), (24, 1),
                                  (31, 0), (32, 0), (32, 1)])
@pytest.mark.parametrize("m,n", SHAPES + [(20000, 7), (5000, 100)])
def test_one_matrix(ccm, m, n, b, sa):
    for bx, sx in X:
        a, x = _rand(m + b, (m, n), b, sa), _rand(n + bx, (n, 1), bx, sx)
        y = ccm.matvec(_pack(ccm, a, b), _pack(ccm, x, bx), capacity=ccm.words_for(m, 1, 64))
        o = _oracle(a, x)
        if o is None:
            assert y.status == ccm.E_OVERFLOW
        else:
            assert_same_packed(y, o, f"{m}x{n} {b}/{sa} x {bx}/{sx}")
