"""Admission by memory: a matmul is served in as little memory as 4 bytes per
field of its operands beside C and its output (host logic; the last test runs it)."""
from types import SimpleNamespace

import numpy as np
import pytest

torch = pytest.importorskip("torch")
ccm = pytest.importorskip("paper_1303_0270_gb300.ccm")
serve = pytest.importorskip("paper_1303_0270_gb300.serve")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1303_0270_gb300 import build
    build.build()


def _up(v, to):
    return (v + to - 1) // to * to


def _four_bytes_per_field(m, k, n):
    """C in int64 and four bytes per field, both operands in whole tiles."""
    return (_up(8 * m * n, 256) + _up(4 * _up(m, 128) * _up(k, 128), 256)
            + _up(4 * _up(n, 64) * _up(k, 128), 256) + 256)


def _server(store, budget):
    srv = serve.Server.__new__(serve.Server)
    srv.store, srv.mem_budget, srv.used = store, budget, 0
    return srv


@pytest.mark.parametrize("m,k,n", [(64, 64, 64), (300, 200, 520), (3001, 2503, 3500),
                                   (8192, 8192, 8192), (2, 8000, 70)])
@pytest.mark.parametrize("b", [3, 12, 16, 20])
def test_matmul_admitted_at_four_bytes_per_field(m, k, n, b):
    store = [SimpleNamespace(rows=r, cols=c, width=b, is_signed=1, capacity=ccm.words_for(r, c, b))
             for r, c in ((m, k), (k, n))]
    r = serve.Request(0, "matmul", 0.0, a=0, b=1)
    out = 4 * ccm.words_for(m, n, ccm.bound_matmul(*store)) + 64
    tight = out + _four_bytes_per_field(m, k, n)
    roomy = out + ccm.workspace_bytes(ccm.OP_MATMUL, m, k, n)
    srv = _server(store, tight)
    assert srv._admit(r) and srv.used == r.nbytes <= tight
    assert r.ws_bytes or roomy <= tight
    assert not srv._admit(serve.Request(1, "matmul", 0.0, a=0, b=1))  # the budget is spent
    assert not _server(store, tight - 1)._admit(r)
    srv = _server(store, roomy)
    assert srv._admit(r) and r.ws_bytes == 0 and srv.used == roomy


@pytest.mark.gpu
@pytest.mark.parametrize("b", [4, 12, 18])
def test_matmul_served_in_a_tight_budget(b):
    import oracle
    import synth
    from gpu_util import assert_same_packed, device, lib_ccm, to_dev
    device()
    lib_ccm()
    m, k, n = 200, 300, 400
    a = synth.uniform_signed(1, 0, m * k, b).reshape(m, k)
    c = synth.uniform_signed(2, 0, k * n, b).reshape(k, n)
    store = [ccm.pack(to_dev(a)), ccm.pack(to_dev(c))]
    resident = sum(4 * (ccm.HEADER_WORDS + p.capacity) for p in store)
    out = 4 * ccm.words_for(m, n, ccm.bound_matmul(*store)) + 64
    srv = serve.Server(store, resident + out + _four_bytes_per_field(m, k, n), streams=2)
    trace = [serve.Request(i, "matmul", 0.0, a=0, b=1) for i in range(3)]
    stats = srv.run(trace)
    assert stats.peak_bytes <= srv.mem_budget and len(stats.latencies) == 3
    o = oracle.matmul(oracle.pack(a), oracle.pack(c))
    for r in trace:
        assert_same_packed(r.out, o, f"served product {b} bits")
    assert np.all([r.ws_bytes for r in trace])
