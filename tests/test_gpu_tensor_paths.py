"""The stored spectrum does not depend on the memory a plan's generation had: the
radial tables, one of them, or neither give the same bytes
(tests/tensor_paths_check.cu), so a served solve equals its plan solved alone."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.mark.gpu
def test_tables_and_points_give_the_same_bytes(tmp_path):
    import __graft_entry__ as g
    lib = g.build()
    from paper_2504_19410_gb300 import build as b
    exe = str(tmp_path / "tensor_paths_check")
    r = subprocess.run([b.nvcc(), *b.ARCH, "-std=c++17", "-I" + b.INCLUDE, os.path.join(HERE, "tensor_paths_check.cu"),
                        lib, "-o", exe, "-Xlinker", "-rpath," + os.path.dirname(lib)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout.strip().splitlines()[-1] == "grids 8 differing 0", out.stdout
