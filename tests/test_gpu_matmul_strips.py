"""A matmul workspace without room for the digit planes of both operands: the
product stays on the tensor cores and goes strip by strip.  Words against the
oracle (integer work: tolerance 0), nothing written past the workspace, and the
launches that tell the path: with the planes whole one launch for them and one for
the product, two more for every further strip."""
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


def _up(v, to):
    return (v + to - 1) // to * to


def _least(m, k, n, b):
    """The least workspace of the explicit tensor path: C in int64, and one byte
    per field and 4 bits of the wider operand's width."""
    w = (b + 3) // 4
    cols = _up(n, 256 if w == 1 else 128 if w == 2 else 64)
    return (_up(8 * m * n, 256) + _up(w * _up(m, 128) * _up(k, 128), 256)
            + _up(w * cols * _up(k, 128), 256) + 256)


def _run(ccm, pa, pb, c, nbytes, path):
    """(launches, intact): the product with a workspace of nbytes and a guard behind it."""
    buf = torch.full((nbytes + 4096,), 0x5A, dtype=torch.uint8, device=device())
    c.buf.zero_()
    before = ccm.launch_count()
    ccm.matmul_into(pa, pb, c, path=path, ws=buf[:nbytes])
    launches = ccm.launch_count() - before
    return launches, bool(torch.all(buf[nbytes:] == 0x5A))


SIZES = [(300, 200, 520), (513, 130, 257), (64, 65, 63), (1000, 257, 90), (129, 64, 1025),
         (2, 300, 700)]


@pytest.mark.parametrize("m,k,n", SIZES)
@pytest.mark.parametrize("ba,sa,bb,sb", [(4, 1, 4, 0), (1, 0, 3, 1), (8, 0, 8, 1), (12, 1, 11, 0),
                                         (16, 0, 16, 1), (12, 0, 2, 1)])
def test_least_workspace_stays_on_the_tensor_cores(ccm, m, k, n, ba, sa, bb, sb):
    a, b = _rand(m + ba, (m, k), ba, sa), _rand(n + bb, (k, n), bb, sb)
    pa, pb = ccm.pack(to_dev(a)), ccm.pack(to_dev(b))
    o = oracle.matmul(oracle.pack(a), oracle.pack(b))
    need = _least(m, k, n, max(ba, bb))
    for bits in (64, 31):  # C in int64 and in int32
        c = ccm.PackedMatrix(m, n, ccm.words_for(m, n, bits))
        whole, _ = _run(ccm, pa, pb, c, ccm.workspace_bytes(ccm.OP_MATMUL, m, k, n),
                        ccm.MATMUL_TENSOR)
        for path in (ccm.MATMUL_TENSOR, ccm.MATMUL_AUTO):
            launches, intact = _run(ccm, pa, pb, c, need, path)
            assert intact
            assert launches >= whole and (launches - whole) % 2 == 0
            if o.width <= bits:
                assert_same_packed(c, o, f"{m}x{k}x{n} {ba}/{sa} x {bb}/{sb}")
            else:
                assert c.status == ccm.E_CAPACITY
    with pytest.raises(ccm.CCMError) as e:
        _run(ccm, pa, pb, c, need - 256, ccm.MATMUL_TENSOR)
    assert e.value.status == ccm.E_CAPACITY


@pytest.mark.parametrize("m,k,n", SIZES[:4])
@pytest.mark.parametrize("ba,bb", [(20, 18), (12, 12), (8, 3)])
def test_every_room_gives_the_same_words(ccm, m, k, n, ba, bb):
    """From hardly any room for planes (the CUDA cores) to more than enough."""
    a, b = _rand(m, (m, k), ba, 1), _rand(n, (k, n), bb, 0)
    pa, pb = ccm.pack(to_dev(a)), ccm.pack(to_dev(b))
    o = oracle.matmul(oracle.pack(a), oracle.pack(b))
    full = ccm.workspace_bytes(ccm.OP_MATMUL, m, k, n)
    least = _least(m, k, n, max(ba, bb)) if ba <= 16 else _up(8 * m * n, 256) + 256
    seen = set()
    for part in (0.0, 0.05, 0.2, 0.35, 0.5, 0.7, 0.9, 1.0):
        c = ccm.PackedMatrix(m, n, ccm.words_for(m, n, 64))
        launches, intact = _run(ccm, pa, pb, c, int(least + part * (full - least)) // 256 * 256,
                                ccm.MATMUL_AUTO)
        assert intact
        assert_same_packed(c, o, f"{m}x{k}x{n} {ba} x {bb}, {part} of the room")
        seen.add(launches)
    if ba > 16:  # the CUDA cores, strips, and the planes whole
        assert len(seen) >= 3
