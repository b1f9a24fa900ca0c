"""Checks that need the kernels' own scratch, as small programs compiled with the library's
sources (tests/native): each returns 0, or prints what is wrong and returns 1."""
import os
import subprocess

import pytest

from paper_2509_26193_gb300 import build

pytestmark = pytest.mark.gpu

NATIVE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native")


def _run(tmp_path, program, sources=()):
    exe = str(tmp_path / "check")
    cmd = [build.nvcc(), *build.ARCH, *build.FLAGS, "--threads", "0", "-I", build.CSRC,
           os.path.join(NATIVE, program), *(os.path.join(build.CSRC, s) for s in sources), "-o",
           exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr


def test_sort_pass_ignores_tickets_past_its_grid(tmp_path):
    _run(tmp_path, "sort_tickets.cu")


def test_noalloc_order_does_not_depend_on_what_its_scratch_holds(tmp_path):
    _run(tmp_path, "noalloc_scratch.cu", ("sort.cu", "scan.cu"))
