"""Output arrays keep their contents while their pages are touched ahead of the
copy back (csrc/bc_pages.h), so a call that fails leaves them as they were
(tests/pages_check.cpp, compiled here with g++)."""
import os
import shutil
import subprocess
import tempfile

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_touching_pages_changes_no_byte():
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "pages_check")
        subprocess.check_call([cxx, "-O2", "-std=c++17", "-pthread", "-o", exe, os.path.join(HERE, "pages_check.cpp")])
        r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
