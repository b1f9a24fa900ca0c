"""The radix sort's tile states (csrc/tile_state.h, compiled for the host) hold every count
and prefix that the library's capacities allow: up to 0x7ffffff0 elements, all of them in
one digit. The look-back over them is replayed here as the kernel does it."""
import ctypes
import shutil
import subprocess

import numpy as np
import pytest

from paper_2509_26193_gb300 import build

SRC = r"""
#include "tile_state.h"
using namespace rl;
extern "C" uint32_t count_state(uint32_t c) { return state_of_count(c); }
extern "C" uint32_t prefix_state(uint32_t p) { return state_of_prefix(p); }
extern "C" int published(uint32_t s) { return state_published(s); }
// the digits before tile n: counts back to the nearest prefix; -1: not published
extern "C" int64_t look_back(const uint32_t *state, int64_t n)
{
    uint32_t words = 0;
    int64_t t = n - 1;
    for (bool done = false; !done; --t) {
        if (!state_published(state[t])) return -1;
        words += state[t];
        done = state_is_prefix(state[t]);
    }
    return state_sum(words, (uint32_t)(n - 1 - t));
}
"""
MOST = 0x7FFFFFF0  # elements a sort may be given
TILE = 4096


@pytest.fixture(scope="module")
def states(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("states")
    (d / "s.cpp").write_text(SRC)
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC,
                    str(d / "s.cpp"), "-o", str(d / "s.so")], check=True)
    L = ctypes.CDLL(str(d / "s.so"))
    L.look_back.restype = ctypes.c_int64
    L.count_state.restype = L.prefix_state.restype = ctypes.c_uint32
    return L


@pytest.mark.parametrize("elements", [0, 1, TILE, (1 << 30) - 1, 1 << 30, (1 << 30) + 5,
                                      MOST - 2 * TILE, MOST])
def test_prefix_of_a_digit_with_every_element(states, elements):
    counts = [TILE, 0, 1, min(TILE, 3)]
    before = max(elements - sum(counts), 0)
    state = np.array([states.prefix_state(before)] + [states.count_state(c) for c in counts],
                     np.uint32)
    assert all(states.published(int(s)) for s in state)
    want = before
    for t in range(1, len(state) + 1):
        assert states.look_back(state.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(t)) == want
        if t <= len(counts):
            want += counts[t - 1]


def test_a_cleared_word_is_not_published(states):
    state = np.array([states.prefix_state(7), 0], np.uint32)
    assert not states.published(0)
    assert states.look_back(state.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(2)) == -1
    assert states.published(states.count_state(0)) and states.published(states.prefix_state(0))
