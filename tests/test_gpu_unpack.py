"""Unpack in runs of 512 fields: every width in both sign modes, sizes at the
edges of a run and of a word, both entry types, and destinations aligned only to
their entries; exact (integer work)."""
import numpy as np
import pytest

import synth
from gpu_util import device, lib_ccm, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b", list(range(1, 33)))
@pytest.mark.parametrize("signed", [0, 1])
def test_unpack_runs(b, signed):
    device()
    ccm = lib_ccm()
    lo, hi = synth.signed_range(b) if signed else (0, (1 << b) - 1)
    for n in (1, 2, 63, 511, 512, 513, 1024, 1025, 5 * 512 + 77):
        v = synth.uniform_int(b + n, 0, n, lo, hi)
        v[0], v[-1] = hi, lo
        p = ccm.PackedMatrix(1, n, ccm.words_for(1, n, b), device())
        ccm.pack_into(to_dev(v.reshape(1, n)), p)
        for dtype in (torch.int64, torch.int32):
            if dtype == torch.int32 and b == 32 and not signed:
                continue
            for skip in (0, 1):  # the destination on and off a 16-byte boundary
                buf = torch.full((n + 2 + skip,), -77, dtype=dtype, device=device())
                out = buf[skip:skip + n].view(1, n)
                assert np.array_equal(ccm.unpack(p, dtype=dtype, out=out).cpu().numpy()[0], v)
                assert torch.all(buf[skip + n:] == -77)  # nothing past the end
