"""The cells of the face kernels' bricks (csrc/dg_brick.cuh, index arithmetic
alone, compiled here for the host): a block reads and writes result rows of
the cells it owns and of no others, every cell is owned once, and the rows
around a brick are the periodic neighbours of its cells.  Meshes below, at and
past a brick (4 x 4 x 2 cells) in every direction."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r'''
#include "dg_brick.cuh"
using dg::sf::Brick;
extern "C" {
int bricks(int N) { return Brick::count(N); }
void own_rows(int N, long* out)
{
    for (int q = 0; q < Brick::count(N); ++q)
        for (int r = 0; r < 32; ++r) out[q * 32 + r] = Brick(q, N).own(r);
}
long cell(int q, int N, int i, int j, int k) { return Brick(q, N).cell(i, j, k); }
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("brick")
    (d / "brick.cpp").write_text(SRC)
    so = str(d / "brick.so")
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2401_06841_gb300", "csrc"), str(d / "brick.cpp"), "-o", so], check=True)
    L = C.CDLL(so)
    L.cell.restype = C.c_long
    return L


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7, 8, 9, 13])
def test_every_cell_is_read_and_written_by_one_block(lib, N):
    nb = lib.bricks(N)
    out = (C.c_long * (32 * nb))()
    lib.own_rows(N, out)
    own = [c for c in out if c >= 0]
    assert all(c >= -1 for c in out)
    assert len(own) == len(set(own)) == N ** 3


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7, 8, 9, 13])
def test_rows_around_a_brick_are_periodic_neighbours(lib, N):
    nb = lib.bricks(N)
    out = (C.c_long * (32 * nb))()
    lib.own_rows(N, out)
    for q in range(nb):
        for r in range(32):
            c = out[q * 32 + r]
            if c < 0:
                continue
            i, j, k = r % 4, (r // 4) % 4, r // 16
            x, y, z = c % N, (c // N) % N, c // (N * N)
            assert lib.cell(q, N, i, j, k) == c
            for d in (-1, 1):
                assert lib.cell(q, N, i + d, j, k) == (z * N + y) * N + (x + d) % N
                assert lib.cell(q, N, i, j + d, k) == (z * N + (y + d) % N) * N + x
                assert lib.cell(q, N, i, j, k + d) == ((z + d) % N * N + y) * N + x
