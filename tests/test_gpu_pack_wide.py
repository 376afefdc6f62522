"""Packs wider than 32 bits beyond the one-launch size (whole words cut from one
or two fields), against the oracle word for word."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import assert_same_packed, device, lib_ccm, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b", list(range(30, 65)))
@pytest.mark.parametrize("signed", [0, 1])
def test_wide_pack(b, signed):
    device()
    ccm = lib_ccm()
    n = 70001  # 68 tiles of 1024 and a ragged one
    lo, hi = synth.signed_range(b) if signed else (0, (1 << min(b, 63)) - 1)
    v = synth.uniform_int(b, 0, n, lo, hi)
    v[0], v[-1] = hi, lo
    v = v.reshape(1, n)
    p = ccm.pack(to_dev(v), capacity=ccm.words_for(1, n, 64))
    assert_same_packed(p, oracle.pack(v), f"wide pack {b}/{signed}")
