"""molora_forward_host enqueues on several streams: in which order, and what a refused launch leaves behind.  csrc/api.cu is linked against
a fake runtime and fake launchers (fake_runtime.cpp) that log every call; nothing runs and no GPU is needed."""
import ctypes
import os
import subprocess
import sys
import threading

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


def call(lib, N, C, shapes, fail=("", -1), priority=0, shared_x=True, stream=STREAM):
    """(status, log) of a gate-routed call; the host buffers lie 1 GB apart."""
    projs = (_HostProjC * len(shapes))(*[_HostProjC((X if shared_x else X + (100 + i << 30)), X + (i + 1 << 30), 0x2000, 0x3000, a, b, r, 1.0)
                                         for i, (a, b, r) in enumerate(shapes)])
    need = lib.molora_forward_host_arena_bytes(projs, len(shapes), M.BF16, N, C, M.ROUTE_GATE, 0)
    assert need > 0
    lib.fake_reset(fail[0].encode(), fail[1], priority)
    st = lib.molora_forward_host(M.ROUTE_GATE, None, None, 0, G, None, 0, projs, len(shapes), M.BF16, N, C, 1 << 45, need, None, stream)
    return st, [(w[0], [int(v) for v in w[1:]]) for w in (line.split() for line in lib.fake_log().decode().splitlines())]


ATTENTION = [(2048, 2048, 16), (2048, 1024, 16), (2048, 1024, 16), (2048, 2048, 16)]
CALLS = [(2048, ATTENTION), (5000, ATTENTION), (2048, [(2048, 512, 32), (2048, 8192, 16)]), (4100, [(4096, 2048, 16)]), (2048, [(2048, 2048, 64), (2048, 8192, 16)]),
         (300, [(1024, 1024, 16)])]
LAUNCHES = ("route", "group", "apply", "apply_pair", "apply_jobs")


def before(log, stream=STREAM):
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
    return sets, last.get(stream, frozenset())


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


def test_a_thread_keeps_one_pair_of_streams(fake):
    """Made by its first call, with the priority of the caller's stream, made again for another priority, given back when the thread ends."""
    def names(log, kind):
        return [a[0] for n, a in log if n == kind]
    logs = []
    def work():
        for priority in (0, 0, -3, -3):
            for N, shapes in ((2048, ATTENTION), (5000, ATTENTION), (4100, [(4096, 2048, 16)])):
                logs.append((priority, call(fake, N, 8, shapes, priority=priority)[1]))
        fake.fake_reset(b"", -1, 0)
    thread = threading.Thread(target=work)
    thread.start()
    thread.join()
    made = [[(a[1], p) for n, a in log if n == "stream"] for p, log in logs]
    assert [len(m) for m in made] == [2] + [0] * 5 + [2] + [0] * 5 and all(q == p for m in made for q, p in m)
    assert sum(len(names(log, "event")) for _, log in logs) <= 2 * (2 + 7 + 4)
    end = [(w[0], [int(v) for v in w[1:]]) for w in (line.split() for line in fake.fake_log().decode().splitlines())]
    for kind in ("stream", "event"):
        assert sorted(sum((names(log, kind) for _, log in logs), [])) == sorted(sum((names(log, "destroy_" + kind) for _, log in logs), names(end, "destroy_" + kind)))


FORKED = """
import ctypes, os, sys
lib = ctypes.CDLL(sys.argv[1])
lib.molora_forward_host_arena_bytes.restype = ctypes.c_size_t
class P(ctypes.Structure):
    _fields_ = [(n, ctypes.c_void_p) for n in ("x", "y", "A", "B")] + [(n, ctypes.c_int32) for n in ("d_in", "d_out", "rank")] + [("scale", ctypes.c_float)]
projs = (P * 2)(*[P(0x10000000, 0x10000000 + (i + 1 << 30), 0x2000, 0x3000, 2048, 2048, 16, 1.0) for i in range(2)])
v, n = ctypes.c_void_p, ctypes.c_int64
need = lib.molora_forward_host_arena_bytes(projs, 2, 1, n(2048), 8, 1, 0)
assert lib.molora_forward_host(1, None, None, 0, v(0x1000), None, 0, projs, 2, 1, n(2048), 8, v(1 << 45), ctypes.c_size_t(need), None, v(0x11)) == 0
lib.fake_report_at_exit()
if os.fork() == 0:
    ctypes.CDLL(None).exit(0)
os.wait()
print("parent", flush=True)
"""


def test_a_forked_child_ends_without_touching_its_parents_streams(fake):
    res = subprocess.run([sys.executable, "-c", FORKED, fake._name], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    child, parent = res.stdout.split("parent")
    assert "end" in child and "destroy_stream" not in child and parent.count("destroy_stream") == 2


def test_calls_of_one_thread_on_two_streams_follow_what_they_read(fake):
    """The second call's work meets the first one's on the kept streams: each caller's stream still follows all of its own."""
    both = []
    for stream in (STREAM, STREAM + 1):
        st, log = call(fake, 2048, 8, ATTENTION, stream=stream)
        assert st == 0
        both += [(n, a, stream) for n, a in log]
    ran, _ = before([(n, a) for n, a, _ in both])
    for stream in (STREAM, STREAM + 1):
        own = {i for i in ran if both[i][2] == stream}
        _, at_end = before([(n, a) for n, a, _ in both], stream)
        assert own <= at_end


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
