"""molora_forward_host enqueues on several streams: in which order, and what a refused launch leaves behind.  csrc/api.cu is linked against
a fake runtime and fake launchers (fake_runtime.cpp) that log every call; nothing runs and no GPU is needed."""
import ctypes
import os
import subprocess

import pytest

import paper_2603_15965_b200 as M
from paper_2603_15965_b200.binding import _HostProjC

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
STREAM, X, G = 0x11, 0x10000000, 0x1000


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    cmd = ["nvcc", "-std=c++17", "-O1", "-cudart", "none", "-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC", "-shared",
           "-Xlinker", "-Bsymbolic", "-I", os.path.join(ROOT, "include"), "-o", out, os.path.join(HERE, "fake_runtime.cpp"),
           os.path.join(ROOT, "paper_2603_15965_b200", "csrc", "api.cu")]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    lib = ctypes.CDLL(out)
    lib.fake_log.restype = ctypes.c_char_p
    lib.molora_forward_host_arena_bytes.restype = ctypes.c_size_t
    lib.molora_forward_host_arena_bytes.argtypes = M.load_library().molora_forward_host_arena_bytes.argtypes
    lib.molora_forward_host.argtypes = M.load_library().molora_forward_host.argtypes
    lib.molora_debug_set.argtypes = [ctypes.c_char_p, ctypes.c_int64]
    return lib


def call(lib, N, C, shapes, fail=("", -1), priority=0, shared_x=True):
    """(status, log) of a gate-routed call; the host buffers lie 1 GB apart."""
    projs = (_HostProjC * len(shapes))(*[_HostProjC((X if shared_x else X + (100 + i << 30)), X + (i + 1 << 30), 0x2000, 0x3000, a, b, r, 1.0)
                                         for i, (a, b, r) in enumerate(shapes)])
    need = lib.molora_forward_host_arena_bytes(projs, len(shapes), M.BF16, N, C, M.ROUTE_GATE, 0)
    assert need > 0
    lib.fake_reset(fail[0].encode(), fail[1], priority)
    st = lib.molora_forward_host(M.ROUTE_GATE, None, None, 0, G, None, 0, projs, len(shapes), M.BF16, N, C, 1 << 45, need, None, STREAM)
    return st, [(w[0], [int(v) for v in w[1:]]) for w in (line.split() for line in lib.fake_log().decode().splitlines())]


ATTENTION = [(2048, 2048, 16), (2048, 1024, 16), (2048, 1024, 16), (2048, 2048, 16)]
CALLS = [(2048, ATTENTION), (5000, ATTENTION), (2048, [(2048, 512, 32), (2048, 8192, 16)]), (4100, [(4096, 2048, 16)]), (2048, [(2048, 2048, 64), (2048, 8192, 16)]),
         (300, [(1024, 1024, 16)])]
LAUNCHES = ("route", "group", "apply", "apply_pair", "apply_jobs")


def before(log):
    """For every entry the set of entries that have run when it runs, from stream order, events and waits; and those the caller's stream
    follows at the end."""
    last, event, sets = {}, {}, {}
    for i, (name, a) in enumerate(log):
        if name == "wait":
            last[a[0]] = last.get(a[0], frozenset()) | event.get(a[1], frozenset())
        elif name == "record":
            event[a[1]] = last.get(a[0], frozenset())
        elif name in ("upload", "download") + LAUNCHES:
            sets[i] = last.get(a[0], frozenset())
            last[a[0]] = sets[i] | {i}
    return sets, last.get(STREAM, frozenset())


@pytest.mark.parametrize("N,shapes", CALLS)
@pytest.mark.parametrize("shared_x", [True, False])
def test_every_step_follows_what_it_reads_and_the_stream_follows_all(fake, N, shapes, shared_x):
    st, log = call(fake, N, 8, shapes, shared_x=shared_x)
    assert st == 0
    ran, at_end = before(log)
    assert at_end == frozenset(ran)
    applies = [(i, a[1], a[3:]) for i, (n, a) in enumerate(log) if n.startswith("apply")]
    route, = [i for i, (n, _) in enumerate(log) if n == "route"]
    for i, rows, projs in applies:
        assert route in ran[i]
        there = [(log[u][1][1], log[u][1][1] + log[u][1][3]) for u in ran[i] if log[u][0] == "upload"]
        for at, cols in zip(projs[0::2], projs[1::2]):       # x and y of every projection: there, whole
            end = at + rows * cols * 2
            while at < end:
                reach = max((hi for lo, hi in there if lo <= at), default=0)
                assert reach > at
                at = reach
    back = 0
    for i, (n, a) in enumerate(log):
        if n == "download":
            back += a[3]
            launch, = [(j, rows * cols * 2) for j, rows, projs in applies for at, cols in zip(projs[2::4], projs[3::4]) if at == a[2]]
            assert launch[0] in ran[i] and launch[1] == a[3]  # ... after the one launch that finishes it
    assert back == sum(N * b * 2 for _, b, _ in shapes)
    for kind in ("stream", "event"):
        made = [a[0] for n, a in log if n == kind]
        assert sorted(made) == sorted(a[0] for n, a in log if n == "destroy_" + kind)


@pytest.mark.parametrize("N,shapes", CALLS)
def test_a_call_that_is_refused_half_way_returns_no_results(fake, N, shapes):
    """Whichever launch, upload or hand-over of the work before the results fails: no copy into any y_host has been enqueued, and the
    caller's stream follows whatever has been."""
    _, whole = call(fake, N, 8, shapes)
    last = max(i for i, (n, _) in enumerate(whole) if n.startswith("apply"))
    for name in LAUNCHES + ("upload", "record"):
        for k in range(sum(n == name for n, _ in whole[: last + 1])):
            st, log = call(fake, N, 8, shapes, fail=(name, k))
            assert st != 0
            assert not any(n == "download" for n, _ in log), (name, k)
            ran, at_end = before(log)
            if name != "record":
                assert at_end == frozenset(ran)


@pytest.mark.parametrize("priority", [0, -3])
def test_streams_of_a_call_have_the_priority_of_the_callers(fake, priority):
    _, log = call(fake, 2048, 8, ATTENTION, priority=priority)
    made = [a[1] for n, a in log if n == "stream"]
    assert len(made) == 2 and set(made) == {priority}


def test_scratch_of_one_projection_spares_the_control_words_of_another(fake):
    """1100 tokens, "small_path" 3: the rank-64 projection on the pair, whose scratch begins where the workspace does when it is applied by
    itself; the rank-16 one in pieces would be small enough for the job-list kernel, whose control words are there."""
    fake.molora_debug_set(b"small_path", 3)
    try:
        st, log = call(fake, 1100, 32, [(1024, 1024, 64), (1024, 8192, 16)])
    finally:
        fake.molora_debug_set(b"small_path", 0)
    assert st == 0
    pair, jobs = ([a[2] for n, a in log if n == name] for name in ("apply_pair", "apply_jobs"))
    assert pair and not set(pair) & set(jobs)
