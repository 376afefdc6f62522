"""Every instance of the tensor matmul's product kernel (tile widths 256, 224, 192,
128 and 64 with 32-bit accumulators, 128 and 64 with 64-bit ones) on sizes that the
rule sends to it, with ragged last tiles, rows and blocks of k.  The rule is asked
with the GPU's own SM count (a small program around matmul_tile.h), so a size that
no longer reaches its instance fails.  Words against the oracle's exact product."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
import synth
from conftest import ROOT

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "matmul_tile.h"
int main(int argc, char** argv) {  // pairs, then m n acc32 ...
  for (int i = 2; i + 2 < argc; i += 3)
    std::printf("%d\n", ccm::tc::tile_columns(strtoull(argv[i], 0, 10), strtoull(argv[i + 1], 0, 10),
                                              atoi(argv[i + 2]) != 0, strtoull(argv[1], 0, 10)));
}
"""

# (columns of the tile, 32-bit accumulators, m, n): ragged in m and n
CASES = [(256, 1, 2049, 2040), (224, 1, 3000, 2500), (192, 1, 2049, 2049), (128, 1, 513, 2500),
         (64, 1, 700, 333), (128, 0, 1025, 2401), (64, 0, 900, 333)]


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("tile")
    (d / "tile.cpp").write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", "-I",
                    os.path.join(ROOT, "paper_1303_0270_gb300", "csrc"), str(d / "tile.cpp"), "-o",
                    str(d / "tile")], check=True)

    def ask(pairs, cases):
        args = [str(v) for acc32, m, n in cases for v in (m, n, acc32)]
        out = subprocess.run([str(d / "tile"), str(pairs), *args], capture_output=True, text=True,
                             check=True).stdout
        return [int(v) for v in out.split()]

    return ask


def test_every_instance_has_a_size(rule):
    """On 152 SMs (76 pairs); also: the widths chosen are the instances'."""
    assert rule(76, [c[1:] for c in CASES]) == [c[0] for c in CASES]
    sizes = [(acc32, m, n) for acc32 in (0, 1) for m in (1, 255, 257, 3001, 40000)
             for n in (1, 65, 500, 4096, 9001)]
    got = rule(76, sizes)
    assert set(got) <= {256, 224, 192, 128, 64}
    assert all(c <= 128 for (acc32, _, _), c in zip(sizes, got) if not acc32)


def _rand(seed, shape, b, signed):
    lo, hi = synth.signed_range(b) if signed else (0, (1 << b) - 1)
    v = synth.uniform_int(seed, 0, int(np.prod(shape)), lo, hi).reshape(shape)
    v.flat[0], v.flat[-1] = hi, lo  # the width is b exactly
    return v


@pytest.mark.gpu
@pytest.mark.parametrize("cols,acc32,m,n", CASES)
@pytest.mark.parametrize("k", [129, 577])  # blocks of 64: an odd number, a ragged last one
def test_instance(rule, cols, acc32, m, n, k):
    from gpu_util import assert_same_packed, device, lib_ccm, to_dev, torch
    device()
    ccm = lib_ccm()
    pairs = torch.cuda.get_device_properties(0).multi_processor_count // 2
    assert rule(pairs, [(acc32, m, n)]) == [cols]
    # one and several digit pairs; a.bits + b.bits + bits of k <= 31 tells the accumulators
    for (ba, sa), (bb, sb) in ((((8, 1), (8, 0)), ((13, 1), (7, 1))) if acc32
                               else (((12, 1), (12, 0)), ((20, 1), (18, 1)))):
        assert (ba + bb + k.bit_length() <= 31) == bool(acc32)
        a, b = _rand(m + ba, (m, k), ba, sa), _rand(n + bb, (k, n), bb, sb)
        c = ccm.matmul(ccm.pack(to_dev(a)), ccm.pack(to_dev(b)), path=ccm.MATMUL_AUTO)
        exact = (a.astype(np.float64) @ b.astype(np.float64)).astype(np.int64)  # sums < 2^53
        assert_same_packed(c, oracle.pack(exact), f"{m}x{k}x{n} {ba} x {bb} bits")
