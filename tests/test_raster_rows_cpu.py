"""The GPU builder's edge walk (csrc/raster.h), compiled for the host, against
geom.h's exact predicates: every grid order, edges one lattice unit high and
2^26 wide among them, whose step of half a row must not be computed (its
quotient does not fit 32 bits)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_edge_walk_equals_geom(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    exe = str(tmp_path / "raster_rows")
    subprocess.run([cxx, "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "raster_rows.cpp")], check=True)
    # half a second; a walk that steps a quotient down by ones takes hours
    p = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert p.returncode == 0, p.stdout
    assert int(p.stdout.split()[0]) > 100_000
