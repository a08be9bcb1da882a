"""Hand-overs between the thread blocks of a one-launch run, and the sums of
their row counts, without a GPU.

csrc/nsli_handover.h says which words an iteration writes and reads.  Here it
is compiled for the host, and the order that the grid's counters give is
followed event by event: a read has to come after the write it is meant to
see, and no other write of the same word may be able to come in between."""
import ctypes
import os
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2003_09956_gb300", "csrc")


@pytest.fixture(scope="module")
def words(tmp_path_factory):
    d = tmp_path_factory.mktemp("handover")
    src = d / "words.cpp"
    src.write_text('#include "nsli_handover.h"\n'
                   'extern "C" int stat_half(int k) { return nsli::stat_half(k); }\n'
                   'extern "C" int dx_half_written(int k) { return nsli::dx_half_written(k); }\n'
                   'extern "C" int dx_half_read(int k) { return nsli::dx_half_read(k); }\n'
                   'extern "C" int iterations_of(long long b) { return nsli::iterations_of(b); }\n'
                   '// 32 lanes added by two 32-bit reductions, as warp_count does\n'
                   'extern "C" long long lanes_total(const long long *h) {\n'
                   '    unsigned int lo = 0, hi = 0;\n'
                   '    for (int i = 0; i < 32; ++i) {\n'
                   '        const nsli::CountParts c = nsli::count_parts(h[i]);\n'
                   '        lo += c.lo;\n'
                   '        hi += c.hi;\n'
                   '    }\n'
                   '    return nsli::count_join(lo, hi);\n'
                   '}\n')
    lib = d / "words.so"
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    return ctypes.CDLL(str(lib))


def run_events(words, columns, iters, modap):
    """The events of every block in program order: (kind, counter, word,
    value).  columns[b]: does block b reduce columns?"""
    out = []
    for b, has in enumerate(columns):
        ev = []
        for k in range(iters):
            ev.append(("write", None, ("stat", b, words.stat_half(k)), k))
            ev += [("arrive", ("A", k), None, None), ("wait", ("A", k), None, None)]
            for c, other in enumerate(columns):
                ev.append(("read", None, ("stat", c, words.stat_half(k)), k))
                if k > 0 and other:
                    ev.append(("read", None, ("dx", c, words.dx_half_read(k)), k - 1))
            if modap:
                if has:
                    ev.append(("arrive", ("C", k), None, None))
                ev.append(("wait", ("C", k), None, None))
            if has:   # a block with several rounds of columns: before B; the last round's: after its arrival
                ev.append(("write", None, ("dx", b, words.dx_half_written(k)), k))
                ev.append(("arrive", ("B", k), None, None))
                ev.append(("write", None, ("dx", b, words.dx_half_written(k)), k))
            ev.append(("wait", ("B", k), None, None))
        out.append(ev)
    return out


def faults(events):
    """Reads that may see another value than the one they are meant to."""
    n = len(events)
    pos = {}   # counter -> [(block, index of its arrival)]
    for b, ev in enumerate(events):
        for i, (kind, cnt, _, _) in enumerate(ev):
            if kind == "arrive":
                pos.setdefault(cnt, []).append((b, i))
    # known[b][i][c]: how many of block c's events are over when event i of
    # block b begins
    known = [[None] * (len(ev) + 1) for ev in events]
    done = [0] * n
    now = [[0] * n for _ in range(n)]
    while any(done[b] < len(events[b]) for b in range(n)):
        moved = False
        for b in range(n):
            while done[b] < len(events[b]):
                kind, cnt, _, _ = events[b][done[b]]
                if kind == "wait":
                    if any(done[c] <= i for c, i in pos.get(cnt, [])):
                        break
                    for c, i in pos[cnt]:
                        now[b] = [max(u, v) for u, v in zip(now[b], known[c][i])]
                        now[b][c] = max(now[b][c], i)
                known[b][done[b]] = list(now[b])
                done[b] += 1
                now[b][b] = done[b]
                moved = True
        assert moved, "a wait that never ends"
    bad = []
    for b, ev in enumerate(events):
        for i, (kind, _, word, value) in enumerate(ev):
            if kind != "read":
                continue
            for c, other in enumerate(events):
                for j, (k2, _, w2, v2) in enumerate(other):
                    if k2 != "write" or w2 != word:
                        continue
                    before = known[b][i][c] > j
                    after = known[c][j][b] > i
                    if v2 <= value and not before or v2 > value and not after:
                        bad.append((word, "read", b, value, "write", c, v2))
    return bad


@pytest.mark.parametrize("modap", [False, True])
@pytest.mark.parametrize("columns", [(True,), (True, True), (True, True, False), (True, False, False)])
def test_no_word_is_overwritten_while_it_may_be_read(words, columns, modap):
    assert faults(run_events(words, columns, 6, modap)) == []


def test_one_half_for_dx_would_be_overwritten(words):
    """The check sees the fault: with a single half, step k's words are
    written while step k - 1's may still be read (ModAP's sum of y^2 holds up
    the blocks that have columns, not those without)."""
    class One:
        stat_half = staticmethod(words.stat_half)
        dx_half_written = staticmethod(lambda k: 0)
        dx_half_read = staticmethod(lambda k: 0)
    for modap, columns in ((False, (True, True)), (False, (True, False)), (True, (True, False))):
        assert faults(run_events(One, columns, 4, modap))


@pytest.mark.parametrize("lanes", [[0] * 32, [1] * 32, [2 ** 26 - 1] * 32, [2 ** 26] * 32, [2 ** 31 - 1] * 32,
                                   [2 ** 31] + [0] * 31, [2 ** 52 + 2 ** 26 - 1] * 32,
                                   [(i * 0x9e3779b97f4a7c15) % 2 ** 40 for i in range(32)]])
def test_counts_of_a_warp_add_exactly(words, lanes):
    """Counts whose total leaves 32 bits (a system of more than 2^31 rows may
    have them all violated; its total is the index of a table)."""
    words.lanes_total.restype = ctypes.c_longlong
    assert words.lanes_total((ctypes.c_longlong * 32)(*lanes)) == sum(lanes)


@pytest.mark.parametrize("log2", [4, 20, 26, 27, 30, 31, 32, 33, 35, 36, 37, 38])
@pytest.mark.parametrize("off", [-16, 0, 16])
def test_a_launch_reads_64_gib_at_most(words, log2, off):
    """... unless one iteration reads more, so that a launch keeps the device
    for some 10 ms."""
    words.iterations_of.argtypes = [ctypes.c_longlong]
    size = max(16, (1 << log2) + off)
    k = words.iterations_of(size)
    assert 1 <= k <= 1024
    assert k == 1 or k * size <= 64 << 30
    assert k == 1024 or (k + 1) * size > 64 << 30    # and no less than that allows
