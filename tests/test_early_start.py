"""When a product may start early behind the library's own producers of sign words and scales (CPU): the note's rule against a brute-force
model, and the source rules that it relies on."""
import ctypes
import os
import random
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_36800_b200", "csrc")

HARNESS = r"""
#include "early_start.h"
using namespace bd;
extern "C" {
void* note_new() { return new ProducerNote; }
void note_delete(void* n) { delete static_cast<ProducerNote*>(n); }
void produced(void* n) { static_cast<ProducerNote*>(n)->produced(); }
void* product_begin(void* n, int device, size_t stream, unsigned long long capture, int known, int enabled, int* early) {
    auto* p = new ProductStart(*static_cast<ProducerNote*>(n), enabled != 0, [&](StreamKey* k) {
        k->device = device; k->stream = reinterpret_cast<const void*>(stream); k->capture = capture;
        return known != 0;
    });
    *early = p->early;
    return p;
}
void product_end(void* p, int launched) {
    auto* s = static_cast<ProductStart*>(p);
    if (launched) s->launched();
    delete s;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("early_start")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-pthread", "-I", CSRC, str(d / "h.cpp"), "-o", str(d / "h.so")], check=True)
    l = ctypes.CDLL(str(d / "h.so"))
    l.note_new.restype = l.product_begin.restype = ctypes.c_void_p
    l.note_delete.argtypes = l.produced.argtypes = [ctypes.c_void_p]
    l.product_begin.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_size_t, ctypes.c_ulonglong, ctypes.c_int, ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    l.product_end.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return l


class Note:
    def __init__(self, lib):
        self.lib, self.n = lib, lib.note_new()

    def produce(self):   # a whole producer call: before its first launch, after its last
        self.lib.produced(self.n)
        self.lib.produced(self.n)

    def begin(self, stream, device=0, capture=0, known=True, enabled=True):
        early = ctypes.c_int()
        p = self.lib.product_begin(self.n, device, stream, capture, known, enabled, ctypes.byref(early))
        return p, bool(early.value)

    def product(self, stream, **kw):
        p, early = self.begin(stream, **kw)
        self.lib.product_end(p, 1)
        return early


A, B = 0x1000, 0x2000


def test_no_producer_no_delay(lib):
    n = Note(lib)
    assert n.product(A) and n.product(B, capture=3) and not n.product(A, enabled=False) and n.product(A)


def test_a_product_elsewhere_does_not_use_the_note_up(lib):
    for other in (dict(stream=B), dict(stream=A, device=1), dict(stream=A, capture=7)):
        n = Note(lib)
        n.produce()                      # on A
        assert not n.product(**other)    # another stream, the same handle on another device, or one that is only recorded
        assert not n.product(A) and n.product(A)
        assert n.product(**other)
        n.produce()
        assert not n.product(A) and not n.product(**other)


def test_capture(lib):
    n = Note(lib)
    n.product(A)
    n.produce()                          # recorded in capture 5
    assert not n.product(B)              # an eager product in between
    assert not n.product(A, capture=5) and n.product(A, capture=5)
    assert not n.product(A, capture=6)   # the next capture knows nothing of this one
    assert not n.product(A) and n.product(A)


def test_what_cannot_be_told_is_not_early_and_not_remembered(lib):
    n = Note(lib)
    assert n.product(A, known=False)     # (no producer yet: not asked)
    n.produce()
    assert not n.product(A, known=False) and not n.product(A, known=False)
    p, early = n.begin(A)                # a launch that fails
    lib.product_end(p, 0)
    assert not early and not n.product(A)
    assert n.product(A)
    assert not n.product(A, enabled=False)


def test_two_threads_on_one_stream(lib):
    # a product between a producer's two marks, and one that begins before another's launch
    n = Note(lib)
    lib.produced(n.n)
    assert not n.product(A)
    lib.produced(n.n)
    assert not n.product(A) and n.product(A)
    n.produce()
    p, early = n.begin(A)
    assert not early and not n.product(A)
    lib.product_end(p, 1)
    assert n.product(A)
    # one that began before a producer and is launched behind it answers nothing
    n.produce()
    p, early = n.begin(A)
    n.produce()
    lib.product_end(p, 1)
    assert not early and not n.product(A)


@pytest.mark.parametrize("seed,keys", [(s, 6) for s in range(6)] + [(s, 900) for s in range(2)])
def test_against_all_of_history(lib, seed, keys):
    # early <=> a product of the same key was launched without the early start, after it had begun behind the last mark of every producer.
    # (With more keys than are held, entries are forgotten: then only =>.)
    rng = random.Random(seed)
    n = Note(lib)
    names = [(rng.randrange(2), 0x100 * (i + 1), rng.choice((0, 0, i + 1))) for i in range(keys)]
    open_products, settled, now, last_mark, early_count = [], {}, 0, 0, 0
    for _ in range(6000 if keys < 100 else 20000):
        now += 1
        what = rng.random()
        if what < (0.15 if keys < 100 else 0.0005):
            lib.produced(n.n)
            last_mark = now
        elif what < 0.4 and open_products:
            p, key, t, early = open_products.pop(rng.randrange(len(open_products)))
            launched = rng.random() < 0.9
            lib.product_end(p, launched)
            if launched and not early and t > last_mark:
                settled[key] = t
        else:
            key = rng.choice(names)
            p, early = n.begin(key[1], device=key[0], capture=key[2])
            allowed = last_mark == 0 or settled.get(key, 0) > last_mark
            assert (early == allowed) if keys < 100 else (allowed or not early)
            early_count += early
            open_products.append((p, key, now, early))
            if len(open_products) > 4:
                p, key, t, early = open_products.pop(0)
                lib.product_end(p, 1)
                if not early and t > last_mark:
                    settled[key] = t
    assert early_count > 100
    for p, *_ in open_products:
        lib.product_end(p, 0)


def test_producers_release_nothing_before_their_results():
    # what is queued behind a producer with an early start must not begin before the results are written: its last kernel never asks for it
    # (compress's first kernel does, for the finishing kernel alone, which waits)
    finish = open(os.path.join(CSRC, "compress.cu")).read()
    finish = finish[finish.index("__global__ void compress_finish_kernel("):]
    finish = re.sub(r"//[^\n]*", "", finish[:finish.index("\n}")])
    assert "grid_launch_dependents" not in finish and finish.index("grid_dependency_wait()") < finish.index("partial[")
    simple = open(os.path.join(CSRC, "kernels_simple.cu")).read()
    pack = simple[simple.index("pack_kernel("):simple.index("unpack_kernel(")]
    assert "launch_dependents" not in pack


def test_every_producer_notes_its_launches():
    api = open(os.path.join(CSRC, "api.cu")).read()
    for launch in ("bd::launch_pack(", "bd::launch_compress("):
        assert api.count(launch) == 1 and re.search(r"const bd::Producing producing\(g_producers\);\s+if \(" + re.escape(launch), api)
    assert len(re.findall(r"bd::ProductStart start\(", api)) == api.count("start.launched();") == 2
