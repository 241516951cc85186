"""The following's 32-bit filter (csrc/abg.cuh) against its 64-bit form on the host, with every signed
overflow trapped (tests/follow_filter_check.cpp).  No GPU."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_narrow_filter_decides_as_the_wide_one_without_signed_overflow(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "follow_filter_check")
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-fsanitize=signed-integer-overflow",
                           "-fsanitize-undefined-trap-on-error",
                           "-I", os.path.join(ROOT, "paper_1712_09434_gb300", "csrc"), "-x", "c++",
                           os.path.join(HERE, "follow_filter_check.cpp"), "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
    out = r.stdout.split()
    assert int(out[1]) > 500000 and int(out[3]) > 1000
