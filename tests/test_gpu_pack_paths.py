"""Which kernel packs a dense matrix hangs on its size, alignment and the output's
capacity.  Every way, on sizes that reach it (up to 65,536 entries: one launch;
beyond: tiles at the width of the capacity, two passes, or run-time widths), int32
and int64, aligned to 16 bytes and to an entry only, with the entry that sets the
width or the sign in the first tile, in the last and nowhere; against the oracle
word for word (integer work: tolerance 0)."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import assert_same_packed, device, lib_ccm, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ccm():
    device()
    return lib_ccm()


def _dev(a, dtype, offset):
    """a on the GPU, `offset` entries into a 16-byte aligned buffer."""
    flat = torch.empty(a.size + offset, dtype=dtype, device=device())
    flat[offset:] = torch.from_numpy(a.ravel()).to(device()).to(dtype)
    return flat[offset:].view(a.shape)


def _narrow(seed, shape, b, signed):
    """Entries of b - 1 bits (b = 1: zeros)."""
    if b == 1:
        return np.zeros(shape, dtype=np.int64)
    lo, hi = synth.signed_range(b - 1) if signed and b > 2 else (0, (1 << (b - 1 - signed)) - 1)
    return synth.uniform_int(seed, 0, int(np.prod(shape)), lo, hi).reshape(shape)


def _place(a, where, b, signed):
    """The one entry that makes the width b and the sign `signed`."""
    v = -(1 << (b - 1)) if signed else (1 << b) - 1
    if where is not None:
        a.flat[where] = v
    return a


def _check(ccm, a, dtype, offset, capacity_width, single_pass=True, what=""):
    rows, cols = a.shape
    m = ccm.PackedMatrix(rows, cols, ccm.words_for(rows, cols, capacity_width) + 64, device())
    m.capacity -= 64
    m.buf.fill_(-1)
    ccm.pack_into(_dev(a, dtype, offset), m, single_pass=single_pass)
    assert_same_packed(m, oracle.pack(a), what)
    assert bool(torch.all(m.buf[ccm.HEADER_WORDS + m.capacity:] == -1)), what


# one launch: CTAs of 512 entries, 8 vectors per thread and step
@pytest.mark.parametrize("n", [1, 2, 3, 5, 31, 511, 512, 513, 4095, 8193, 16385, 32770, 49153, 65533,
                               65534, 65535, 65536])
@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
@pytest.mark.parametrize("offset", [0, 1])
def test_one_launch(ccm, n, dtype, offset):
    for b, signed in ((1, 0), (9, 1), (31, 0), (32, 1)) + (((45, 0), (64, 1)) if dtype == torch.int64
                                                         else ()):
        for where in {0, n // 2, n - 1}:  # (the only entry that sets width or sign)
            a = _place(_narrow(n + b, (1, n), b, signed), where, b, signed)
            _check(ccm, a, dtype, offset, max(b, 1), what=f"{n} at {b}/{signed}, entry {where}")


SHAPE = (131, 1003)  # 131,393 entries: 129 tiles of 1024, the last one ragged


@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
@pytest.mark.parametrize("b", [1, 5, 8, 13, 16, 21, 31, 32])
@pytest.mark.parametrize("signed", [0, 1])
def test_beyond_one_launch(ccm, dtype, b, signed):
    if dtype == torch.int32 and b == 32 and not signed:
        pytest.skip("no unsigned 32-bit entries in int32")
    n = SHAPE[0] * SHAPE[1]
    for where in (0, n // 2, n - 1, None):  # the first tile, one inside, the last, no entry
        a = _place(_narrow(b, SHAPE, b, signed), where, b, signed)
        what = f"{b}/{signed} in {dtype}, entry {where}"
        _check(ccm, a, dtype, 0, b, what=what + ", tiles")
        _check(ccm, a, dtype, 0, min(b + 2, 32), what=what + ", tiles re-coded")
        _check(ccm, a, dtype, 0, b, single_pass=False, what=what + ", two passes")
        _check(ccm, a, dtype, 1, b, what=what + ", aligned to an entry")
        _check(ccm, a, dtype, 0, 64, what=what + ", run-time width")
        _check(ccm, a, dtype, 1, 64, what=what + ", run-time width, aligned to an entry")


def test_too_small_an_output(ccm):
    for n in (65536, 131393):
        a = _place(_narrow(3, (1, n), 12, 0), n - 1, 12, 0)
        m = ccm.PackedMatrix(1, n, ccm.words_for(1, n, 12), device())
        m.capacity = ccm.words_for(1, n, 11)
        m.buf.fill_(-1)
        ccm.pack_into(_dev(a, torch.int64, 0), m)
        assert m.status == ccm.E_CAPACITY
        assert bool(torch.all(m.buf[ccm.HEADER_WORDS + m.capacity:] == -1))
