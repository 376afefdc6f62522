"""The matvec of rows that begin anywhere in a word: every width in both sign
modes, x as one and as two byte digits and as int32, rows shorter and longer
than a warp's 32 segments, sizes at the edges of segments and stages, and the
one-launch pack of y at its limit, against the oracle word for word (integer
work: tolerance 0)."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import assert_same_packed, device, lib_ccm, to_dev

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


def _check(ccm, m, n, ba, sa, bx, sx):
    a, x = _rand(m + ba, (m, n), ba, sa), _rand(n + bx, (n, 1), bx, sx)
    y = ccm.matvec(_pack(ccm, a, ba), _pack(ccm, x, bx), capacity=ccm.words_for(m, 1, 64))
    try:
        o = oracle.matvec(oracle.pack(a), oracle.pack(x))
    except OverflowError:  # (the widest pairs pass int64)
        assert y.status == ccm.E_OVERFLOW
        return
    assert_same_packed(y, o, f"{m}x{n} {ba}/{sa} x {bx}/{sx}")


@pytest.mark.parametrize("b", list(range(1, 33)))
@pytest.mark.parametrize("sa", [0, 1])
def test_every_width(ccm, b, sa):
    for bx, sx in [(8, 1), (7, 0), (8, 0), (14, 1), (14, 0), (15, 1), (24, 0)]:
        _check(ccm, 37, 1100, b, sa, bx, sx)


@pytest.mark.parametrize("m,n", [(1, 65), (3, 33), (500, 97), (1, 5000), (130, 1023), (130, 1025),
                                 (64, 1280), (9, 8192), (2, 70001)])
@pytest.mark.parametrize("ba,sa", [(5, 0), (14, 1), (16, 1), (32, 0)])
def test_edges_of_rows_and_stages(ccm, m, n, ba, sa):
    for bx, sx in [(8, 1), (12, 1), (20, 0)]:
        _check(ccm, m, n, ba, sa, bx, sx)


@pytest.mark.parametrize("m", [16385, 65536, 65537])
def test_one_launch_pack_of_y(ccm, m):
    _check(ccm, m, 33, 9, 1, 8, 1)


def test_two_products_in_one_chain(ccm):
    """y = A x + B z with rows of different lengths, widths and routes."""
    m = 300
    a, x = _rand(1, (m, 701), 11, 1), _rand(2, (701, 1), 8, 1)
    b, z = _rand(3, (m, 95), 20, 0), _rand(4, (95, 1), 18, 1)
    y = ccm.matvec2(_pack(ccm, a, 11), _pack(ccm, x, 8), _pack(ccm, b, 20), _pack(ccm, z, 18))
    assert_same_packed(y, oracle.pack(a @ x + b @ z), "matvec2")


def test_invalid_operand_is_reported(ccm):
    a, x = _rand(5, (50, 77), 9, 1), _rand(6, (77, 1), 8, 1)
    pa, px = _pack(ccm, a, 9), _pack(ccm, x, 8)
    px.buf[0] = 0  # not a packed matrix
    y = ccm.matvec_into(pa, px, ccm.PackedMatrix(50, 1, ccm.words_for(50, 1, 64), device()))
    assert y.status == ccm.E_INPUT
