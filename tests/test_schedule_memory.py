"""The context's device copies of its schedules, against a CUDA runtime that is a few host functions (tests/fake_cuda.cpp):
which streams and how much memory a context takes, and what a call's kernels find there.  Needs no GPU."""
import ctypes
import os
import subprocess

import pytest

from paper_2604_24432_b200 import binding as ksa
from paper_2604_24432_b200 import build as ksa_build

HERE = os.path.dirname(os.path.abspath(__file__))


class Counts(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("streams_made", "streams_gone", "mallocs", "frees", "device_syncs", "uploads_default", "uploads_own")]


def _run(*cmd):
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, (cmd, r.stderr[-2000:])
    return r.stdout


def _symbols(obj, *nm_flags):
    return {line.split()[-1] for line in _run("nm", *nm_flags, obj).splitlines() if line.strip()}


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    """The library's host object linked with the fake runtime; what neither defines is a function that returns zero."""
    ksa_build.build()
    d = str(tmp_path_factory.mktemp("fake"))
    host, obj, lib = os.path.join(ksa_build.OBJ_DIR, "ksa_api.o"), os.path.join(d, "fake.o"), os.path.join(d, "libfake.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(ksa_build._nvcc())) or "/usr/local/cuda", "include")
    _run("g++", "-std=c++17", "-O1", "-fPIC", "-I" + cuda, "-c", os.path.join(HERE, "fake_cuda.cpp"), "-o", obj)
    missing = (_symbols(host, "-u") | _symbols(obj, "-u")) - _symbols(obj, "--defined-only")
    missing = sorted(s for s in missing if s.startswith(("cuda", "__cuda", "_ZN3ksa")))
    with open(os.path.join(d, "stubs.s"), "w") as f:
        f.write(".text\n" + "".join(".globl %s\n.type %s, @function\n%s:\n" % (s, s, s) for s in missing) + "xorl %eax, %eax\nret\n.section .note.GNU-stack,\"\",@progbits\n")
    _run("g++", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-o", lib, host, obj, os.path.join(d, "stubs.s"))
    L = ctypes.CDLL(lib)
    L.fake_counts.restype = Counts
    L.fake_seqs.restype = ctypes.c_void_p
    L.fake_capture.argtypes = L.fake_graph_destroy.argtypes = [ctypes.c_void_p]
    L.fake_seqs_text.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return L


class FakeContext:
    def __init__(self, L):
        self.L, self.handle, self.before = L, ctypes.c_void_p(), L.fake_counts()
        assert L.ksa_create(ctypes.byref(self.handle), 0) == ksa.KSA_OK

    def count(self, name):
        return getattr(self.L.fake_counts(), name) - getattr(self.before, name)

    def call(self, lens, Hq=4, stream=None):
        """ksa_qkv_prepare, whose launch reads the schedule's device copy; returns where that copy stands."""
        prob = ksa.Problem(lens, 8, 1, 16, Hq, Hq, 64, 0.125)
        p, buf = prob.params(), ctypes.c_void_p(1 << 20)
        rc = self.L.ksa_qkv_prepare(self.handle, *[buf] * 9, ctypes.c_float(0.5), ctypes.c_float(1e4), 0, ctypes.byref(p), ctypes.c_void_p(stream))
        assert rc == ksa.KSA_OK, rc
        at = self.L.fake_seqs()
        assert self.text(at, len(lens)) == list(lens)
        return at

    def text(self, at, n):
        return [self.L.fake_seqs_text(at, i) for i in range(n)]

    def close(self):
        assert self.L.ksa_destroy(self.handle) == ksa.KSA_OK


def test_the_upload_stream_is_made_once_and_shared(fake):
    """A context that uploads no schedule (one that decodes) takes no stream; the others share one, which goes with the last of
    them.  No upload waits for the default stream."""
    a, b, c = (FakeContext(fake) for _ in range(3))
    assert a.count("streams_made") == 0
    for i in range(5):
        for ctx in (a, b):
            ctx.call([64 + i])
            ctx.call([64 + i])
    assert a.count("streams_made") == 1 and a.count("uploads_own") == 10 and a.count("uploads_default") == 0
    assert a.count("device_syncs") == 0
    a.close()
    c.close()
    b.call([9])
    assert a.count("streams_gone") == 0
    b.close()
    assert a.count("streams_gone") == 1 and a.count("streams_made") == 1 and a.count("mallocs") == a.count("frees")


def test_a_full_arena_waits_once_and_starts_over(fake):
    c = FakeContext(fake)
    at = [c.call([4096 + 8 * i], Hq=16) for i in range(40)]                      # some 10 KB each, 256 KB in all
    assert len(set(at)) < len(at)                                                # parts are used again ...
    assert 1 <= c.count("device_syncs") <= 4                                     # ... after the device has been waited for
    c.close()
    assert c.count("mallocs") == c.count("frees")


@pytest.mark.parametrize("n", [4096, 70_000])                                    # schedules of 10 KB, and larger than the arena
def test_a_graph_keeps_the_schedule_it_was_recorded_with(fake, n):
    """A call recorded into a graph reads its schedule at every replay: the context's later calls, however many, leave that
    memory alone until the graph is gone, and then take it back."""
    c = FakeContext(fake)
    kept = {}
    for graph in (1, 2, 3):
        lens = [n + 8 * graph, 77]
        at = c.call(lens, Hq=16)
        fake.fake_capture(graph)
        assert c.call(lens, Hq=16) == at
        fake.fake_capture(None)
        kept[graph] = (at, ctypes.string_at(at, 8192))
    def others(count):
        for i in range(count):
            c.call([n + 1000 + 8 * i], Hq=16)
            c.call([64 + i, 5], Hq=2)
            for at, was in kept.values():
                assert ctypes.string_at(at, 8192) == was
    others(40)
    assert c.count("device_syncs") > 0                                           # the arena did go round
    for graph in (2, 1, 3):
        fake.fake_graph_destroy(graph)
        del kept[graph]
        others(20)
    assert c.count("mallocs") - c.count("frees") <= 3                            # status word, arena, one block to be freed next
    c.close()
    assert c.count("mallocs") == c.count("frees")


def test_a_graph_may_outlive_its_context(fake):
    c = FakeContext(fake)
    c.call([500])
    fake.fake_capture(9)
    c.call([500])
    fake.fake_capture(None)
    c.close()
    assert c.count("mallocs") == c.count("frees")
    fake.fake_graph_destroy(9)
