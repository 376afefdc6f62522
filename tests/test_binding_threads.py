"""Every call has argument structs of its own: what one thread's call reads does
not change when another thread changes the same matrix object and makes a call
with it (a fake library records what it is given; no GPU needed)."""
import copy
import ctypes
import pickle
import threading
from types import SimpleNamespace

import pytest

torch = pytest.importorskip("torch")
ccm = pytest.importorskip("paper_1303_0270_gb300.ccm")

STREAM = SimpleNamespace(cuda_stream=0)


def _fields(ref):
    m = ctypes.cast(ref, ctypes.POINTER(ccm.Matrix)).contents
    return m.hdr, m.words, m.capacity, m.rows, m.cols


@pytest.mark.parametrize("shared", [0, 1, 2])
def test_a_call_keeps_its_arguments(monkeypatch, shared):
    mats = [ccm.PackedMatrix(8, 4, 64, "cpu") for _ in range(3)]
    held, other = mats[shared], [ccm.PackedMatrix(8, 4, 64, "cpu") for _ in range(3)]
    inside, changed = threading.Event(), threading.Event()
    seen = []

    def add(a, b, c, ws, ws_bytes, stream):
        refs = (a, b, c)
        if not inside.is_set():  # the first call: held inside the library
            before = [_fields(r) for r in refs]
            inside.set()
            assert changed.wait(30)
            seen.append((before, [_fields(r) for r in refs]))
        return ccm.OK

    monkeypatch.setattr(ccm, "lib", lambda: SimpleNamespace(ccm_add=add))
    first = threading.Thread(target=ccm.add_into, args=(*mats, STREAM))
    first.start()
    assert inside.wait(30)
    held.buf = torch.empty(4096, dtype=torch.int32)
    held.capacity = 4000
    other[shared] = held
    ccm.add_into(*other, stream=STREAM)
    changed.set()
    first.join(30)
    (before, after), = seen
    assert before == after


def test_arguments_follow_the_object_and_copies_stand_alone(monkeypatch):
    seen = []
    monkeypatch.setattr(ccm, "lib", lambda: SimpleNamespace(
        ccm_scale=lambda a, s, c, ws, n, st: seen.append((_fields(a), _fields(c))) or ccm.OK))
    a, c = ccm.PackedMatrix(3, 5, 16, "cpu"), ccm.PackedMatrix(3, 5, 32, "cpu")
    ccm.scale_into(a, 7, c, stream=STREAM)
    for make in (copy.copy, copy.deepcopy, lambda m: pickle.loads(pickle.dumps(m))):
        d = make(c)
        d.capacity = 24
        ccm.scale_into(a, 7, d, stream=STREAM)
        assert seen[-1][0] == (a.hdr_ptr, a.words_ptr, 16, 3, 5)
        assert seen[-1][1] == (d.hdr_ptr, d.words_ptr, 24, 3, 5)
        ccm.scale_into(a, 7, c, stream=STREAM)
        assert seen[-1][1] == (c.hdr_ptr, c.words_ptr, 32, 3, 5)
