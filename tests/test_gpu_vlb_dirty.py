"""The variable-length encoder writes every word of its stream whatever the buffer
held before: into words of all ones, through the C entry point, with a guard
behind the stream and one behind the index; words against the oracle."""
import ctypes

import numpy as np
import pytest

import oracle
import synth
from gpu_util import device, lib_ccm, to_dev, torch

pytestmark = pytest.mark.gpu

GUARD = 64


@pytest.mark.parametrize("case", ["word_ends", "mixed", "ones", "wide"])
@pytest.mark.parametrize("n", [1, 7, 64, 1023, 1024, 1025, 2048, 5000, 70001])
def test_stream_over_a_buffer_of_ones(case, n):
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
    o = oracle.vlb_pack(a.reshape(1, n))
    words = len(o.words)
    entries = int(ccm.lib().ccm_vlb_index_entries(1, n))
    dense = to_dev(a)
    ws = torch.full((max(ccm.workspace_bytes(ccm.OP_VLB, 1, n, 0), 256),), 255, dtype=torch.uint8,
                    device=device())
    for fill in (-1, 0x55555555):
        buf = torch.full((ccm.HEADER_WORDS + words + GUARD,), fill, dtype=torch.int32,
                         device=device())
        index = torch.full((entries + GUARD,), fill, dtype=torch.int64, device=device())
        at = buf.data_ptr()
        st = ccm.lib().ccm_vlb_pack(dense.data_ptr(), ccm.I64, 1, n, at, at + 4 * ccm.HEADER_WORDS,
                                    words, index.data_ptr(), ws.data_ptr(), ws.numel(),
                                    ccm._stream(None))
        assert st == ccm.OK
        h = ccm.Header()
        assert ccm.lib().ccm_header_read(at, ctypes.byref(h), ccm._stream(None)) == ccm.OK
        assert (h.status, h.nwords) == (0, words)
        got = buf[ccm.HEADER_WORDS:].cpu().numpy()
        assert np.array_equal(got[:words].view(np.uint32), o.words), (case, n)
        assert np.all(got[words:] == fill) and bool(torch.all(index[entries:] == fill))
