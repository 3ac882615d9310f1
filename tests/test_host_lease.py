"""The pool of page-locked buffers that calls borrow (csrc/host_lease.h), against a stand-in
for the CUDA calls it makes: compiled and run on the CPU."""
import os
import shutil
import subprocess

import pytest

from paper_2603_13618_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def _checks(tmp_path, defines=()):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))),
                           "include")
    exe = str(tmp_path / "host_lease")
    r = subprocess.run([cxx, "-std=c++17", "-pthread", "-I", include, "-I", build.CSRC, *defines,
                        os.path.join(HERE, "host_lease_driver.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stderr
    return dict(line.split(": ") for line in out.stdout.splitlines())


def test_buffers_are_handed_on_only_when_nothing_uses_them(tmp_path):
    checks = _checks(tmp_path)
    assert len(checks) >= 6 and set(checks.values()) == {"ok"}, checks


def test_the_pool_is_bounded_and_calls_beyond_it_make_and_free_no_memory(tmp_path):
    checks = _checks(tmp_path)
    for r in range(3):
        assert checks[f"no buffer is lent twice ({r})"] == "ok", checks
    assert checks["calls beyond the pool's size make and free no memory"] == "ok", checks
    assert checks["kept buffers need no new memory"] == "ok", checks
