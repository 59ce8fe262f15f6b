"""csrc/umma_split.cuh: the cluster size that is chosen on a B200 (clusters that are resident at once as the runtime reports them), for calls
where the choice for one load is a bad one for another (no GPU)."""
import ctypes
import os
import subprocess

import pytest

import paper_2603_15965_b200 as M

CSRC = os.path.join(os.path.dirname(M.__file__), "csrc")
CLUSTERS = [0, 148, 74, 45, 33, 26, 22, 15, 15]
WRAPPER = """
#include "umma_split.cuh"
using namespace molora;
extern "C" int plan(const double* chunks, int nproj, int min_kx, long N, int C, int max_split, const int* clusters)
{
    const UmmaPlan p = choose_umma_split(chunks, nproj, min_kx, N, C, max_split, 148, [&](int s) { return clusters[s]; });
    return p.split * 1000 + p.tile_rows;
}
extern "C" long tiles(long N, int C, int rows, int equal) { return equal ? umma_tiles(N, C, rows).equal : umma_tiles(N, C, rows).uneven; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("split")
    src, out = str(d / "wrapper.cpp"), str(d / "libsplit.so")
    with open(src, "w") as f:
        f.write(WRAPPER)
    cmd = [os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", "-I", CSRC, "-I", os.path.join(os.path.dirname(CSRC), "..", "include"),
           src, "-o", out]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    lib = ctypes.CDLL(out)
    lib.plan.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_long, ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    lib.tiles.argtypes, lib.tiles.restype = [ctypes.c_long, ctypes.c_int, ctypes.c_int, ctypes.c_int], ctypes.c_long
    return lib


def plan(lib, N, C, shapes, max_split=8):
    chunks = (ctypes.c_double * len(shapes))(*[(a + b) // 64 for a, b in shapes])
    return divmod(lib.plan(chunks, len(shapes), min(a for a, _ in shapes) // 64, N, C, max_split, (ctypes.c_int * 9)(*CLUSTERS)), 1000)


def attention(h):
    return [(h, h), (h, h // 4), (h, h // 4), (h, h)]


@pytest.mark.parametrize("N,C,shapes,split", [
    # four projections 2048 wide: an even load has 16 tiles, 64 of 74 clusters of two; an uneven one is thought to have 23
    (1700, 16, attention(2048), 2),
    # an uneven load of 25 and 27: not on the 26 clusters of five
    (3000, 2, [(2048, 2048)], 4), (3000, 4, [(2048, 2048)], 4),
    # few tiles: clusters of eight; many: none
    (1000, 8, [(4096, 4096)], 8), (8192, 16, [(4096, 4096)] * 4, 1),
])
def test_choice(lib, N, C, shapes, split):
    assert plan(lib, N, C, shapes)[0] == split


@pytest.mark.parametrize("N,C,width,tiles", [(2300, 8, 2048, 24), (2300, 8, 4096, 24), (2300, 16, 2048, 32), (2300, 16, 4096, 32), (1000, 16, 2048, 16)])
def test_even_load_stays_in_one_wave(lib, N, C, width, tiles):
    """Segments that all round up: N / 128 + C / 2 tiles fit the next larger clusters, these do not (1.5 to 1.7 times the time)."""
    split, rows = plan(lib, N, C, [(width, width)])
    assert split > 1 and lib.tiles(N, C, 128, 1) == tiles and lib.tiles(N, C, rows, 1) <= CLUSTERS[split]


def test_choice_is_within_the_limits(lib):
    for C in (1, 3, 16, 64):
        for N in (1, 100, 1000, 4000, 20000):
            for shapes in ([(256, 256)], [(512, 64)], attention(1024), [(4096, 12288)]):
                for most in (4, 8):
                    s, rows = plan(lib, N, C, shapes, most)
                    assert 1 <= s <= most and rows in (64, 96, 128) and (s == 1 or min(a for a, _ in shapes) // 64 // s >= 4)
            assert lib.tiles(N, C, 128, 1) >= -(-N // 128) and lib.tiles(N, C, 128, 0) >= C
