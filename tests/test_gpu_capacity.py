"""A product whose exact width needs more words than its output has is reported
and writes nothing past the output's words."""
import numpy as np
import pytest

import synth
from gpu_util import device, lib_ccm, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width", [9, 17])
def test_matmul_result_past_its_capacity(width):
    device()
    ccm = lib_ccm()
    m, k, n = 96, 200, 80
    a = synth.uniform_signed(1, 0, m * k, 8).reshape(m, k)
    b = synth.uniform_signed(2, 0, k * n, 8).reshape(k, n)
    pa, pb = ccm.pack(to_dev(a)), ccm.pack(to_dev(b))
    c = ccm.PackedMatrix(m, n, ccm.words_for(m, n, 32), device())
    c.capacity = ccm.words_for(m, n, width)  # the rest of the buffer is a guard
    c.buf.fill_(0x5A5A5A5A)
    ccm.matmul_into(pa, pb, c)
    assert c.status == ccm.E_CAPACITY
    guard = c.buf[ccm.HEADER_WORDS + c.capacity:]
    assert bool(torch.all(guard == 0x5A5A5A5A))
    assert np.array_equal(ccm.unpack(pa).cpu().numpy(), a)
