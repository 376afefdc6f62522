"""The variable-length encoder at its edges: blocks that end on a word (their
last word has no neighbour), entries of one to 63 bits side by side, inputs
aligned only to their entries, int32 inputs, and more blocks than one step of the
offset scan; against the oracle word for word, or by the round trip."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import device, lib_ccm, to_dev, torch, words_np

pytestmark = pytest.mark.gpu


def _same(v, a):
    o = oracle.vlb_pack(a)
    assert np.array_equal(words_np(v), o.words)


@pytest.mark.parametrize("case", ["word_ends", "mixed", "ones", "wide"])
@pytest.mark.parametrize("n", [1, 64, 1023, 1024, 1025, 5000])
def test_blocks(case, n):
    device()
    ccm = lib_ccm()
    if case == "word_ends":  # every entry 2 + 2 bits: a block is 128 words
        a = np.full(n, 2, dtype=np.int64)
    elif case == "ones":
        a = synth.uniform_int(1, 0, n, 0, 1)
    elif case == "wide":
        a = synth.uniform_int(2, 0, n, 1 << 62, (1 << 63) - 1)
    else:
        a = synth.uniform_int(3, 0, n, 0, (1 << 62)) >> synth.uniform_int(4, 0, n, 0, 62)
    a = a.reshape(1, n)
    dev = to_dev(a)
    _same(ccm.vlb_pack(dev), a)
    # (a dirty buffer, and an input off its 16-byte boundary)
    buf = torch.empty(n + 1, dtype=torch.int64, device=device())
    buf[1:] = dev.view(-1)
    _same(ccm.vlb_pack(buf[1:].view(1, n)), a)
    if a.max() < (1 << 31):
        _same(ccm.vlb_pack(dev.to(torch.int32)), a)


def test_many_blocks_round_trip():
    device()
    ccm = lib_ccm()
    n = 16 * 1024 * 1024 + 4 * 1024 + 5  # more blocks than one step of the scan
    g = torch.Generator(device=device())
    g.manual_seed(7)
    a = torch.randint(0, 1 << 20, (1, n), generator=g, device=device(), dtype=torch.int64)
    a >>= torch.randint(0, 20, (1, n), generator=g, device=device(), dtype=torch.int64)
    v = ccm.vlb_pack(a)
    assert torch.equal(ccm.vlb_unpack(v), a)
