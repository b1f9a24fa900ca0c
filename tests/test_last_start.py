"""The draw's search for its block of ranges (csrc/last_start.h, compiled for the host) finds
the last start at or before the target, as a scan over all starts does, although starts
formed by a shuffle scan in FP64 may fall by a rounding from one to the next."""
import ctypes
import shutil
import subprocess

import numpy as np
import pytest

from paper_2509_26193_gb300 import build

SRC = r"""
#include "last_start.h"
extern "C" int find(const double *start, int nb, double tgt) { return rl::last_start(start, nb, tgt); }
"""


@pytest.fixture(scope="module")
def find(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("starts")
    (d / "s.cpp").write_text(SRC)
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC,
                    str(d / "s.cpp"), "-o", str(d / "s.so")], check=True)
    L = ctypes.CDLL(str(d / "s.so"))
    return lambda start, nb, tgt: L.find(start.ctypes.data_as(ctypes.c_void_p), nb,
                                         ctypes.c_double(tgt))


def _starts(blk):
    """The kernel's exclusive warp scan of 32 block sums."""
    s = np.concatenate([[0.0], blk[:31]])
    for o in (1, 2, 4, 8, 16):
        s = s + np.concatenate([np.zeros(o), s[:-o]])
    return s


@pytest.mark.parametrize("spread", [1.0, 12.0, 40.0])
def test_last_start_at_or_before_the_target(find, spread):
    rng = np.random.default_rng(int(spread))
    falling = 0
    for trial in range(400):
        blk = 2.0 ** (-spread * rng.random(32)) * rng.random(32)
        blk[rng.random(32) < 0.3] = 0.0
        nb = int(rng.integers(1, 33))
        s = _starts(blk)
        falling += int((np.diff(s[:nb]) < 0).any())
        targets = np.concatenate([s[:nb], np.nextafter(s[:nb], 0.0), np.nextafter(s[:nb], 9e9),
                                  rng.random(8) * s[nb - 1], [0.0]])
        for t in targets:
            at = np.nonzero(s[:nb] <= t)[0]
            assert find(s, nb, t) == (at[-1] if len(at) else 0)
    if spread > 1.0:
        assert falling > 0  # the case that a plain bisection gets wrong is among them
