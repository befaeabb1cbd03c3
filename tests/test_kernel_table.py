"""CPU checks of the kernel table that a context fills for its device: each table asks about every
kernel again, keeps refusals, and no launcher keeps an answer of its own outside it."""
import ctypes
import os
import re

from paper_2606_07878_gb300 import still

CSRC = os.path.join(os.path.dirname(still.LIB_PATH), "csrc")
SET = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_int)
ASK = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.POINTER(ctypes.c_int), ctypes.c_void_p, ctypes.c_int)
ROOM = 512


def _table(sms, set_smem, resident):
    """[(status, {cluster size: resident})] of a table filled from these answers."""
    out = (ctypes.c_int32 * (9 * ROOM))()

    def ask(n, fn, size):
        got = resident(fn, size)
        n[0] = got or 0
        return 0 if got is not None else 1

    n = still.lib().still_internal_kernel_table(sms, SET(set_smem), ASK(ask), out, ROOM)
    assert 0 < n <= ROOM
    return [(out[9 * i], {c: out[9 * i + c] for c in range(2, 9)}) for i in range(n)]


def test_every_device_is_asked_about_every_kernel():
    asked = {}

    def device(name, per_size):
        asked[name] = []
        set_smem = lambda fn, b: asked[name].append((fn, b)) or 0  # noqa: E731
        return _table(100, set_smem, lambda fn, size: per_size // size)

    a, b = device("a", 96), device("b", 40)
    assert sorted(asked["a"]) == sorted(asked["b"])  # the second device is set up as the first
    assert len({fn for fn, _ in asked["a"]}) == len(a)  # each kernel once
    pairs = {k for k in range(len(a)) if a[k][1][2]}
    assert len(pairs) >= 20
    for k in pairs:
        assert a[k][1][2] == 48 and b[k][1][2] == 20
    assert any(a[k][1][8] == 12 and b[k][1][8] == 5 for k in pairs)


def test_refused_queries_are_kept_per_kernel():
    bad = set()

    def set_smem(fn, nbytes):
        if not bad:
            bad.add(fn)
        return 1 if fn in bad else 0

    t = _table(152, set_smem, lambda fn, size: None if size == 3 else 1000)
    assert sum(status != 0 for status, _ in t) == 1
    for status, clusters in t:
        assert clusters[3] == 0
        for size in range(2, 9):  # never more than the SMs hold
            assert clusters[size] <= 152 // size
            assert status == 0 or clusters[size] == 0


def test_no_launcher_keeps_state():
    """Function-local statics of the sources: the entry point of the driver, the thread's flag of an
    allocation-free call, names and the list of kernels. (The stand-ins of these tests follow the
    line that introduces them.)"""
    allowed = ("fn = nullptr", "std::once_flag once", "v = false", "names[", "entries")
    found = []
    for name in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, name)).read().split("// Host-only views of the library")[0]
        for line in src.splitlines():
            if re.match(r"\s+static (?!constexpr|inline|__device__)\S+ [^(]*(;|=)", line):
                if not any(a in line for a in allowed):
                    found.append((name, line.strip()))
    assert not found, found
