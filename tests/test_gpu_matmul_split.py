"""The tensor-core matmul's digit splits: every digit count and run length,
operands of different widths and signs, sizes at the edges of tiles and of
blocks of k, against the oracle word for word (integer work: tolerance 0), and
against the CUDA-core path where the split path takes over from it."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import assert_same_packed, device, lib_ccm, to_dev, words_np

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


# (width, signed) pairs: one digit each, 1 x 2, 2 x 1, 2 x 2, 1 x 3, 2 x 3, 3 x 3 digits
WIDTHS = [(1, 0, 1, 1), (8, 0, 8, 0), (9, 1, 8, 1), (12, 1, 5, 1), (12, 1, 12, 1), (11, 0, 11, 0),
          (16, 0, 4, 0), (16, 1, 16, 1), (16, 0, 16, 0), (12, 1, 17, 1), (20, 1, 18, 1),
          (18, 0, 20, 0), (24, 1, 24, 1), (26, 0, 26, 0), (31, 0, 3, 1)]


@pytest.mark.parametrize("ba,sa,bb,sb", WIDTHS)
@pytest.mark.parametrize("m,k,n", [(64, 65, 66), (255, 257, 63), (257, 64, 225), (129, 639, 130)])
def test_splits_against_oracle(ccm, m, k, n, ba, sa, bb, sb):
    a, b = _rand(m + ba, (m, k), ba, sa), _rand(n + bb, (k, n), bb, sb)
    pa, pb = ccm.pack(to_dev(a)), ccm.pack(to_dev(b))
    o = oracle.matmul(oracle.pack(a), oracle.pack(b))
    c = ccm.matmul(pa, pb)
    assert_same_packed(c, o, f"matmul {m}x{k}x{n} {ba}/{sa} x {bb}/{sb}")
    cc = ccm.matmul(pa, pb, path=ccm.MATMUL_CUDACORE)
    assert np.array_equal(words_np(c), words_np(cc))


@pytest.mark.parametrize("ba,sa,bb,sb", [w for w in WIDTHS if w[0] > 1])
def test_largest_sums_over_many_runs(ccm, ba, sa, bb, sb):
    """Entries at the ends of the ranges over several runs of k: the sums that
    the fp32 accumulators must hold exactly are at their largest (all of one
    sign, alternating, and off by one in places)."""
    m, k, n = 130, 2500, 70
    a = np.full((m, k), (1 << (ba - 1)) - 1 if sa else (1 << ba) - 1, dtype=np.int64)
    b = np.full((k, n), (1 << (bb - 1)) - 1 if sb else (1 << bb) - 1, dtype=np.int64)
    a[1::2] = -(1 << (ba - 1)) if sa else 0
    b[:, 1::3] = -(1 << (bb - 1)) if sb else 1
    a[2::4, ::3] ^= 1
    b[5::7] ^= 1
    pa, pb = ccm.pack(to_dev(a)), ccm.pack(to_dev(b))
    c = ccm.matmul(pa, pb)
    try:
        o = oracle.pack(oracle.matmul_dense(a, b))
    except OverflowError:  # (26 x 26 bits unsigned: past int64)
        assert c.status == ccm.E_OVERFLOW
        return
    assert_same_packed(c, o, f"{ba}/{sa} x {bb}/{sb}")


@pytest.mark.parametrize("ba,bb", [(8, 8), (20, 18)])
def test_small_capacity_and_small_workspace(ccm, ba, bb):
    """A result that does not fit its capacity is reported, and a workspace
    without room for the planes still gives the product."""
    import torch
    m, k, n = 96, 200, 80
    a, b = _rand(1, (m, k), ba, 1), _rand(2, (k, n), bb, 1)
    pa, pb = ccm.pack(to_dev(a)), ccm.pack(to_dev(b))
    assert ccm.matmul(pa, pb, capacity=ccm.words_for(m, n, 9)).status == ccm.E_CAPACITY
    o = oracle.matmul(oracle.pack(a), oracle.pack(b))
    c = ccm.PackedMatrix(m, n, ccm.words_for(m, n, 64))
    # (8 bits: the least workspace accepted; 20 bits: C's scratch alone)
    need = m * n * 8 + 256 + (2 * 128 * 256 + 2 * 128 * 256 if ba == 8 else 0)
    ws = torch.empty(need, dtype=torch.uint8, device=device())
    ccm.matmul_into(pa, pb, c, ws=ws)
    assert_same_packed(c, o, "small workspace")


def test_tensor_path_takes_the_least_workspace(ccm):
    """The explicit tensor path accepts every workspace that holds C and a byte
    per field and 4-bit digit, also without room for the planes."""
    import torch
    m, k, n = 128, 200, 256
    a, b = _rand(3, (m, k), 4, 1), _rand(4, (k, n), 4, 1)
    pa, pb = ccm.pack(to_dev(a)), ccm.pack(to_dev(b))
    ws = torch.empty(m * n * 8 + 256 + 128 * 256 + 256 * 256, dtype=torch.uint8, device=device())
    c = ccm.PackedMatrix(m, n, ccm.words_for(m, n, 64))
    ccm.matmul_into(pa, pb, c, path=ccm.MATMUL_TENSOR, ws=ws)
    assert_same_packed(c, oracle.matmul(oracle.pack(a), oracle.pack(b)), "least workspace")
