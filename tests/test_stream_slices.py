"""csrc/stream_slices.cuh: the busiest cluster against a walk over every item, and what the choice costs the host (no GPU)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import paper_2603_15965_b200 as M

CSRC = os.path.join(os.path.dirname(M.__file__), "csrc")
WRAPPER = """
#include <chrono>
#include "stream_slices.cuh"
using namespace molora;
static SliceShapes shapes(int P, const int* in, const int* out)
{
    SliceShapes sh;
    sh.P = P;
    for (int i = 0; i < P; ++i) sh.in[i] = in[i], sh.out[i] = out[i];
    return sh;
}
extern "C" int slices(int P, const int* in, const int* out, long most, int* och, int* ustart) { return slice_outputs(shapes(P, in, out), most, och, ustart); }
extern "C" int busiest(int P, const int* in, const int* out, const int* och, const int* ustart, int clusters, int tiles)
{
    return busiest_cluster(shapes(P, in, out), och, ustart, clusters, tiles);
}
extern "C" int balanced(int P, const int* in, const int* out, int clusters, int tiles, int equal, int* och, int* ustart)
{
    return balanced_units(shapes(P, in, out), clusters, tiles, equal, och, ustart);
}
extern "C" double shortest_us(int P, const int* in, const int* out, int clusters, int tiles)
{
    int och[MOLORA_MAX_PROJECTIONS], ustart[MOLORA_MAX_PROJECTIONS + 1];
    volatile int sink = 0;
    double best = 1e9;
    for (int i = 0; i < 2000; ++i) {
        const auto t0 = std::chrono::steady_clock::now();
        sink = sink + balanced_units(shapes(P, in, out), clusters, tiles, tiles + 4, och, ustart);
        best = std::min(best, std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - t0).count());
    }
    return best;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("slices")
    src, out = str(d / "wrapper.cpp"), str(d / "libslices.so")
    with open(src, "w") as f:
        f.write(WRAPPER)
    cmd = [os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", "-I", CSRC, "-I", os.path.join(os.path.dirname(CSRC), "..", "include"),
           src, "-o", out]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    lib = ctypes.CDLL(out)
    lib.shortest_us.restype = ctypes.c_double
    lib.slices.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_long, ctypes.c_void_p, ctypes.c_void_p]
    return lib


def ints(v):
    return (ctypes.c_int * len(v))(*v)


def walk(ins, outs, och, ustart, clusters, tiles):
    """The same, item by item, as the kernel deals them."""
    load, item = np.zeros(clusters, dtype=np.int64), 0
    for p in range(len(ins)):
        for u in range(ustart[p], ustart[p + 1]):
            cost = 13 * ins[p] + 20 * min(och[p], outs[p] - (u - ustart[p]) * och[p]) + 8
            for _ in range(tiles):
                rnd, c = divmod(item, clusters)
                load[clusters - 1 - c if rnd & 1 else c] += cost
                item += 1
    return int(load.max())


@pytest.mark.parametrize("clusters", [1, 5, 132, 148, 256])
def test_busiest_cluster_and_choice(lib, clusters):
    rng = np.random.default_rng(clusters)
    for _ in range(60):
        P = int(rng.integers(1, 9))
        ins, outs = [int(v) for v in rng.integers(1, 13, P)], [int(v) for v in rng.integers(1, 25, P)]
        tiles = int(rng.choice([1, 2, clusters - 1, clusters, clusters + 1, int(rng.integers(1, 3 * clusters + 2))])) or 1
        equal = int(rng.choice([tiles, max(1, tiles // 2), int(rng.integers(1, 3 * clusters + 2))]))
        och, ustart = (ctypes.c_int * 8)(), (ctypes.c_int * 9)()
        best, best_units, slices_of = None, None, {}
        for most in range(P, P + 5):
            if lib.slices(P, ints(ins), ints(outs), most, och, ustart) < most:
                break
            slices_of[most] = list(och[:P])
            longest = walk(ins, outs, och, ustart, clusters, tiles)
            assert lib.busiest(P, ints(ins), ints(outs), och, ustart, clusters, tiles) == longest
            evenly = walk(ins, outs, och, ustart, clusters, equal)
            if best is None or (longest * 100 < best[0] * 97 and evenly <= best[1]):
                best, best_units = (longest, evenly), most
        assert lib.balanced(P, ints(ins), ints(outs), clusters, tiles, equal, och, ustart) == best_units
        assert list(och[:P]) == slices_of[best_units]


def test_cost_does_not_grow_with_the_tiles(lib):
    """A layer of seven projections: a walk over the items took eight times as long for eight times the tiles (5.7 us for 56 of them)."""
    ins, outs = ints([2, 2, 6, 2, 2, 2, 2]), ints([6, 6, 2, 2, 2, 1, 1])
    few, many = (min(lib.shortest_us(7, ins, outs, 148, t) for _ in range(3)) for t in (14, 112))
    print(few, many)
    assert many < 3 * few


@pytest.mark.parametrize("hidden,chunk,tiles,equal", [(3072, 1024, 20, 32), (2560, 1024, 18, 32), (512, 256, 21, 32)])
def test_no_cut_that_lengthens_an_evenly_spread_load(lib, hidden, chunk, tiles, equal):
    """Layers of few tokens of 32 adapters: a cut that pays for the tiles that are expected would cost the tiles of an even load more."""
    kv, inter = hidden // 4 // 64 * 64, 3 * hidden
    widths = [(hidden, inter), (hidden, inter), (inter, hidden), (hidden, hidden), (hidden, hidden), (hidden, kv), (hidden, kv)]
    ins, outs = ([-(-w[i] // chunk) for w in widths] for i in (0, 1))
    och, ustart = (ctypes.c_int * 8)(), (ctypes.c_int * 9)()
    units = lib.balanced(7, ints(ins), ints(outs), 148, tiles, equal, och, ustart)
    assert walk(ins, outs, och, ustart, 148, equal) <= walk(ins, outs, outs, list(range(8)), 148, equal)
    assert units == 7 and lib.balanced(7, ints(ins), ints(outs), 148, tiles, tiles, och, ustart) > 7
