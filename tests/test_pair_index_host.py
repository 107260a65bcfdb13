"""Index arithmetic of the pair sums' cotangent table (csrc/psum_index.h) on the CPU: for
every boundary length, tile, target and lane the index lies in the table, and for the
lanes that hold a node it is the difference of the two nodes mod M."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2108_01786_gb300", "csrc", "psum_index.h")


@pytest.fixture(scope="module")
def index(tmp_path_factory):
    d = tmp_path_factory.mktemp("psum")
    src, so = str(d / "i.cpp"), str(d / "i.so")
    with open(src, "w") as f:
        f.write(f'#include "{HEADER}"\n'
                'extern "C" int up(int a, int p, int n, int M) { return psum_index_up(a, p, n, M); }\n'
                'extern "C" int down(int a, int p, int n, int M) { return psum_index_down(a, p, n, M); }\n')
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-o", so, src], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("M", [8, 9, 15, 16, 17, 31, 32, 33, 40, 63, 65])
def test_every_lane_reads_its_table(index, M):
    for l0 in range(0, M, 32):                      # tiles of the boundary
        n = min(32, M - l0)
        for im in range(M):                         # targets on the same boundary
            for p in range(32):                     # lanes: p and p + 16 of the pair walk
                up = index.up((l0 - im) % M, p, n, M)
                down = index.down((im - l0) % M, p, n, M)
                assert 0 <= up < M and 0 <= down < M
                if p < n:
                    assert up == (l0 + p - im) % M and down == (im - l0 - p) % M
