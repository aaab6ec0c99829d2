"""What tenom_rhs_noalloc keeps on every GPU that loads the library: the face scratch that the header
names and the face lists, and no second buffer of that size (no GPU)."""
import subprocess

import pytest


def test_static_scratch_is_the_faces_and_their_lists(tmp_path):
    from paper_2010_13289_gb300 import build as B
    obj = tmp_path / "noalloc.o"
    r = subprocess.run([B.nvcc()] + B.ARCH + ["-std=c++17", "-O0", "-I", B.INCLUDE, "-I", B.CSRC, "-c",
                                              B.CSRC + "/tenom_noalloc.cu", "-o", str(obj)], capture_output=True, text=True)
    if r.returncode != 0:
        pytest.fail("nvcc failed:\n" + r.stderr[-3000:])
    # the array's host-side stand-in has its size
    sizes = [int(line.split()[1], 16) for line in
             subprocess.run(["nm", "-S", str(obj)], capture_output=True, text=True).stdout.splitlines()
             if "g_noalloc_scratch" in line and len(line.split()) == 4]
    assert sizes == [(16 + 4) << 20]
