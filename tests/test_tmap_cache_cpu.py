"""The cache of encoded tensor maps (csrc/tmap_cache.h, compiled here with the host compiler and a counting
encoder): the maps of stacks of converted layers all hit from the second pass on, every lookup gives the map
of its own key through evictions and from several threads, and a failed encoding keeps nothing."""
import ctypes
import pathlib
import random
import shutil
import subprocess
import threading

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2606_28516_gb300" / "csrc"
SRC = """
#include "tmap_cache.h"
struct alignas(64) Map { long long v[16]; };
static cm::TmapCache<Map> g_big;
static cm::TmapCache<Map, 64> g_small;
template <class C> long long look(C& c, long long base, long long rows, long long cols, int br, int bc, int el, long long* misses) {
    Map m;
    const int rc = c.get(&m, cm::TmapKey{(const void*)base, rows, cols, br, bc, el}, [&](Map* o) {
        if (base < 0) return -7;
        ++*misses;
        for (auto& x : o->v) x = ((((base * 31 + rows) * 31 + cols) * 31 + br) * 31 + bc) * 31 + el;
        return 0;
    });
    for (auto& x : m.v) if (!rc && x != m.v[0]) return -1;
    return rc ? rc : m.v[0];
}
extern "C" long long big(long long b, long long r, long long c, int br, int bc, int e, long long* n) { return look(g_big, b, r, c, br, bc, e, n); }
extern "C" long long small(long long b, long long r, long long c, int br, int bc, int e, long long* n) { return look(g_small, b, r, c, br, bc, e, n); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    t = tmp_path_factory.mktemp("tmap")
    (t / "t.cpp").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-pthread", "-I", str(CSRC), "-o", str(t / "t.so"),
                    str(t / "t.cpp")], check=True)
    L = ctypes.CDLL(str(t / "t.so"))
    for f in (L.big, L.small):
        f.argtypes = [ctypes.c_longlong] * 3 + [ctypes.c_int] * 3 + [ctypes.POINTER(ctypes.c_longlong)]
        f.restype = ctypes.c_longlong
    return L


def _value(k):
    v = 0
    for x in k:
        v = v * 31 + x
    return (v + 2 ** 63) % 2 ** 64 - 2 ** 63


def _look(f, k):
    n = ctypes.c_longlong(0)
    assert f(*k, ctypes.byref(n)) == _value(k)
    return n.value


def _stack(layers, E, T, d, r, base=1 << 40):
    """The keys of one pass, in order: dense and converted layers in turn, weights one behind another."""
    H, keys, a = 4 * d, [], base
    x, y, z, t = 0x7f0000000000, 0x7f0001000000, 0x7f0002000000, 0x7f0003000000

    def weight(rows, cols, bn, half=True):
        nonlocal a
        keys.append((a, rows, cols, bn // 2, 0, 2))
        if half:
            keys.append((a, rows, cols, bn // 4, 0, 2))
        a += rows * cols * 2

    for l in range(layers):
        if l % 2 == 0:
            keys.append((x, T, d, 128, 0, 2))
            weight(H, d, 128)
            keys.append((z, T, H, 128, 0, 2))
            weight(d, H, 128)
        else:
            keys += [(x, T, d, 8, 4, 2), (a, E, d, 16, 0, 2)]
            a += E * d * 2
            keys.append((x, T, d, 128, 0, 2))
            weight(H, d, 128)
            keys.append((z, T, H, 128, 0, 2))
            weight(r, H, 128)
            keys += [(t, T, r, 128, 0, 2), (z, T, H, 128, 0, 2)]
            weight(d, r, 128)
            for _ in range(E):
                weight(d, H, 128)
        x, y = y, x
    return keys


@pytest.mark.parametrize("layers,E", [(4, 12), (6, 8), (12, 8), (24, 15)])
def test_a_stack_hits_from_its_second_pass_on(lib, layers, E):
    keys = _stack(layers, E, 197, 768, 128, base=(layers * 100 + E) << 40)
    first = sum(_look(lib.big, k) for k in keys)
    assert first >= len(set(keys)) - 8  # x, y, z and t may be there from a stack before
    assert sum(_look(lib.big, k) for k in keys) == 0
    assert sum(_look(lib.big, k) for k in keys) == 0


def test_right_map_through_evictions_and_threads(lib):
    keys = [(i << 8, i % 7, 64, 128, i % 3, 2) for i in range(1, 200)]

    def work(seed, out):
        rng = random.Random(seed)
        try:
            for _ in range(5000):
                _look(lib.small, rng.choice(keys))
            out.append(True)
        except AssertionError:
            out.append(False)

    done = []
    ts = [threading.Thread(target=work, args=(s, done)) for s in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert done == [True] * 4
    new = [((1 << 30) + (i << 8), 5, 64, 128, 0, 2) for i in range(64)]
    assert sum(_look(lib.small, k) for k in new) == 64  # the 64 newest are all there
    assert sum(_look(lib.small, k) for k in new) == 0


def test_failed_encoding_is_passed_on_and_not_kept(lib):
    n = ctypes.c_longlong(0)
    for _ in range(2):
        assert lib.big(-16, 1, 64, 128, 0, 2, ctypes.byref(n)) == -7
    assert n.value == 0
