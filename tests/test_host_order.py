"""Order of the work that the library's host code enqueues: its translation units are linked against a CUDA runtime
that records the calls instead of running them, and what one stream does is checked to be ordered before what
another stream does with the same memory."""
import ctypes
import glob
import os
import subprocess
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from paper_2003_13493_gb300 import build, vio

HERE = os.path.dirname(os.path.abspath(__file__))
OUT = os.path.join(HERE, "_build")


def build_host_library():
    """The library's host code over the fake runtime (device code is compiled but never runs)."""
    lib = os.path.join(OUT, "libvio_host.so")
    sources = sorted(glob.glob(os.path.join(build.CSRC, "*.cu")) + glob.glob(os.path.join(HERE, "fake_cuda", "*.c*")))
    deps = sources + glob.glob(os.path.join(build.CSRC, "*.*h")) + glob.glob(os.path.join(build.INCLUDE, "*.h"))
    if os.path.exists(lib) and all(os.path.getmtime(p) < os.path.getmtime(lib) for p in deps):
        return lib
    os.makedirs(OUT, exist_ok=True)
    tag = f".{os.getpid()}"
    objs = [os.path.join(OUT, os.path.basename(s) + tag + ".o") for s in sources]
    flags = ["-gencode", "arch=compute_103a,code=compute_103a", "-Ofc", "max", "-std=c++17", "-Xcompiler", "-fPIC",
             "-I", build.INCLUDE]
    try:
        with ThreadPoolExecutor(len(sources)) as ex:
            list(ex.map(lambda so: subprocess.check_call([build.nvcc(), *flags, "-c", "-o", so[1], so[0]]),
                        zip(sources, objs)))
        # symbols are bound inside: another CUDA runtime may be loaded in this process
        subprocess.check_call([build.nvcc(), "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", "-o", lib + tag,
                               *objs])
        os.replace(lib + tag, lib)
    finally:
        for o in objs:
            if os.path.exists(o):
                os.remove(o)
    return lib


class Host:
    """A context over the fake runtime."""

    def __init__(self, lib, **cfg):
        self.lib = lib
        self.keep = []
        c = vio.Config()
        lib.vio_config_default(ctypes.byref(c))
        for k, v in cfg.items():
            setattr(c, k, v)
        self.ctx = ctypes.c_void_p()
        assert lib.vio_create(ctypes.byref(self.ctx), ctypes.byref(c)) == 0

    def close(self):
        self.lib.vio_destroy(self.ctx)

    def _call(self, fn, sizes, stream, levels, host, align, cell, extra=()):
        n, lib = len(sizes), self.lib
        room = [((w + 15) // 16 * 16 if align else w | 1) for w, _ in sizes]
        frames = [np.zeros(p * h + 64, np.uint8) for p, (_, h) in zip(room, sizes)]
        outs = [np.full((vio.num_cells(w, h, cell) + 1, 4), 7, np.int32) for w, h in sizes for _ in range(extra and 2 or 1)]
        counts = np.zeros(2 * n, np.int32)
        self.keep += [frames, outs, counts]
        up = lambda a: a.ctypes.data + (-a.ctypes.data) % 16
        if host == "pinned":
            for a in outs:
                lib.fake_pin(ctypes.c_void_p(a.ctypes.data), ctypes.c_size_t(a.nbytes))
        P = ctypes.c_void_p
        dims = (vio.Dims * n)(*[vio.Dims(w, h, p) for p, (w, h) in zip(room, sizes)])
        return fn(self.ctx, (P * n)(*[up(f) + (0 if align else 1) for f in frames]), dims, n, *extra or (15, 9), cell,
                  levels, (P * len(outs))(*[up(o) for o in outs]), P(counts.ctypes.data), P(stream))

    def detect(self, sizes, stream, levels=3, align=True, cell=32):
        return self._call(self.lib.vio_detect, sizes, stream, levels, None, align, cell)

    def detect_host(self, sizes, stream, levels=3, cell=32, out="pinned"):
        return self._call(self.lib.vio_detect_host, sizes, stream, levels, out, True, cell)

    def sweep(self, sizes, stream, levels=3, align=True, cell=32):
        two = ctypes.c_int * 2
        return self._call(self.lib.vio_detect_sweep, sizes, stream, levels, None, align, cell,
                          (two(10, 20), two(9, 9), 2))

    def log(self, clear=False):
        text = self.lib.fake_log().decode()
        if clear:
            self.lib.fake_clear()
        return [line.split() for line in text.splitlines()]


@pytest.fixture(scope="session")
def host_lib():
    path = build_host_library()
    with pytest.MonkeyPatch.context() as m:
        m.setattr(vio, "_lib", None)
        m.setattr(vio, "lib_path", lambda: path)
        return vio.load(build_if_missing=False)


@pytest.fixture
def host(host_lib):
    made = []
    host_lib.fake_log.restype = ctypes.c_char_p
    host_lib.fake_fail.argtypes = [ctypes.c_char_p, ctypes.c_int]
    host_lib.fake_capturing.argtypes = [ctypes.c_void_p, ctypes.c_int]
    host_lib.fake_clear()

    def make(**cfg):
        made.append(Host(host_lib, **cfg))
        return made[-1]

    yield make
    host_lib.fake_capturing(None, 0)
    for h in made:
        h.close()


def ordered(log, first, then):
    """Whether entry `first` is complete before entry `then` can begin: by their stream, by events, or because the
    host waited in between."""
    done = {first}                  # entries that are known to follow `first`
    streams, events, host = {log[first][1]}, set(), False
    for i in range(first + 1, then + 1):
        op, s = log[i][0], log[i][1]
        if host or s in streams:
            done.add(i)
            streams.add(s)
        if op == "record":
            (events.add if s in streams else events.discard)(log[i][2])
        elif op == "wait" and log[i][2] in events:
            streams.add(s)
        elif op == "device_sync" or (op == "stream_sync" and s in streams) or \
                (op == "event_sync" and log[i][2] in events):
            host = True
    return then in done


def covers(entry, address):
    return int(entry[2], 16) <= address < int(entry[2], 16) + int(entry[-1])


S1, S2 = 0x1110, 0x2220  # two non-blocking streams of a caller


def test_the_order_check_itself():
    log = [line.split() for line in ("memset legacy 0x1 8", "launch 0xa k", "record legacy 0xe", "wait 0xb 0xe",
                                     "launch 0xb k", "record 0xb 0xe", "stream_sync 0xb", "launch 0xa k")]
    assert not ordered(log, 0, 1) and ordered(log, 0, 4) and ordered(log, 0, 7)
    assert not ordered(log, 1, 4) and ordered(log, 1, 7)


@pytest.mark.parametrize("sizes", [[(752, 480)], [(1920, 1080)] * 20], ids=["tiles", "persistent"])
def test_cleared_buffers_are_ready_on_any_stream(host, sizes):
    """The cell keys and the kernels' counters are zero before the first kernel of any stream can see them: a fresh
    context's first call, and a call that needs more keys, on another stream."""
    h = host(max_frames=64)
    assert h.detect(sizes, S1) == 0
    assert h.detect(sizes * 3, S2) == 0
    log = h.log()
    launches = {s: next(i for i, e in enumerate(log) if e[0] == "launch" and int(e[1], 16) == s) for s in (S1, S2)}
    clears = [i for i, e in enumerate(log) if e[0] == "memset"]
    assert len(clears) == 3
    for c in clears:
        for s, first in launches.items():
            if c < first:
                assert ordered(log, c, first), (log[c], hex(s))
    assert max(clears[:2]) < launches[S1] < clears[2] < launches[S2]


@pytest.mark.parametrize("small", [[(640, 480)], [(160, 120)] * 70], ids=["tiles", "persistent"])
def test_a_clear_outlives_the_call_that_asked_for_it(host, small):
    """A call that grows the keys and then fails has enqueued nothing that a later call, on another stream, could wait
    for but the clear itself."""
    large = [(1920, 1080)] * 60

    def attempt(budget):
        h = host(max_frames=128, mem_budget_bytes=budget)
        h.log(clear=True)
        return h, h.detect(large, S1)

    lo, hi = 1 << 20, 256 << 20  # the smallest budget that works
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if attempt(mid)[1] == 0 else (mid, hi)
    h, status = attempt(lo - 65536)  # the keys fit, the pyramid does not
    clear = next(i for i, e in enumerate(h.log()) if e[0] == "memset")
    assert status == 2 and not [e for e in h.log() if e[0] == "launch"]
    assert h.detect(small, S2) == 0
    log = h.log()
    assert ordered(log, clear, next(i for i, e in enumerate(log) if e[0] == "launch"))


@pytest.mark.parametrize("before", ["sweep", "detect"])
@pytest.mark.parametrize("sizes", [[(640, 480)], [(1920, 1080)] * 4], ids=["one copy", "groups"])
def test_an_upload_waits_for_the_frames_staged_before_it(host, before, sizes):
    """Unaligned device frames and host frames share the context's input buffer: a host call's copies follow the
    kernels of an earlier call on another stream that read it."""
    h = host(max_frames=64)
    unaligned = [(1921, 1081)] * 30
    assert h.detect_host([(1920, 1080)] * 32, S2) == 0  # the buffer is large enough from here on
    h.log(clear=True)
    if before == "sweep":
        assert h.sweep(unaligned, S1, align=False) == 0
    else:
        assert h.detect(unaligned, S1, align=False) == 0
    assert h.detect_host(sizes, S2) == 0
    log = h.log()
    assert not [e for e in log if e[0] == "malloc" and int(e[3]) > 4 << 20]
    launch = max(i for i, e in enumerate(log) if e[0] == "launch" and int(e[1], 16) == S1)
    copies = [i for i, e in enumerate(log) if e[0] == "copy" and i > launch and int(e[4]) > 200_000]
    assert copies
    for c in copies:
        assert ordered(log, launch, c), log[c]


@pytest.mark.parametrize("op,nth", [("launch", 3), ("launch", 5), ("copy", 3)])
def test_a_grouped_call_that_fails_leaves_nothing_in_flight(host, op, nth):
    """The caller of a synchronous call may free its buffers when it returns, also with an error: no kernel of an
    earlier group still writes records, and no copy still reads frames."""
    h = host(max_frames=64)
    sizes = [(1280, 720)] * 24
    assert h.detect_host(sizes, S1) == 0
    h.log(clear=True)
    h.lib.fake_fail(op.encode(), nth)
    assert h.detect_host(sizes, S1) == 3
    log = h.log(clear=True)
    work = [i for i, e in enumerate(log) if e[0] in ("launch", "copy")]
    assert [e for e in log if e[0] == "launch"] and len({log[i][1] for i in work}) == 2
    end = len(log)
    for i in work:
        assert ordered(log + [["host", "-"]], i, end), log[i]
    assert h.detect_host(sizes, S1) == 0


def test_a_grouped_call_over_the_budget_starts_nothing(host):
    """Every buffer that any group needs is there before the first group begins, so a budget that is too small by
    the keys of a late, larger group is found before any work is enqueued."""
    small, large = [(1280, 720)] * 12, [(3840, 2160)] * 3

    def attempt(budget):
        h = host(max_frames=64, mem_budget_bytes=budget)
        h.log(clear=True)
        return h.detect_host(small + large, S1, cell=32), h.log(clear=True)

    lo, hi = 1 << 20, 256 << 20  # the smallest budget that works
    while hi - lo > 256:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if attempt(mid)[0] == 0 else (mid, hi)
    for budget in (lo, lo - 4096, lo - 65536):
        status, log = attempt(budget)
        assert status == 2 and not [e for e in log if e[0] in ("launch", "copy")], budget


@pytest.mark.parametrize("sizes,align", [([(752, 480)], True), ([(1280, 720)] * 16, True), ([(641, 480)] * 4, False)])
def test_a_captured_stream_takes_the_persistent_kernels(host, sizes, align):
    """Inside a caller's stream capture a detection is refused: a graph replayed later would use resident buffers
    that have been given back when a larger call grew them.  The kernels of small calls are no way around that."""
    h = host(max_frames=64)
    for _ in range(2):
        assert h.detect(sizes, S1, align=align) == 0
    assert any("tile_detect" in e[2] for e in h.log(clear=True) if e[0] == "launch")
    h.lib.fake_capturing(S1, 1)
    assert h.detect(sizes, S1, align=align) == 3
    assert not [e for e in h.log() if e[0] == "launch"]
    h.lib.fake_capturing(None, 0)
    assert h.detect(sizes, S1, align=align) == 0
