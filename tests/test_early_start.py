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
void produced(void* n, int known, unsigned long long capture) { static_cast<ProducerNote*>(n)->produced(known != 0, capture); }
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
    l.note_delete.argtypes = [ctypes.c_void_p]
    l.produced.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_ulonglong]
    l.product_begin.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_size_t, ctypes.c_ulonglong, ctypes.c_int, ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    l.product_end.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return l


class Note:
    def __init__(self, lib):
        self.lib, self.n = lib, lib.note_new()

    def mark(self, capture=0, known=True):
        self.lib.produced(self.n, known, capture)

    def produce(self, **kw):   # a whole producer call: before its first launch, after its last
        self.mark(**kw)
        self.mark(**kw)

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
    for other in (dict(stream=B), dict(stream=A, device=1)):
        n = Note(lib)
        n.produce()                      # on A
        assert not n.product(**other)    # another stream, or the same handle on another device
        assert not n.product(A) and n.product(A)
        assert n.product(**other)
        n.produce()
        assert not n.product(A) and not n.product(**other)


def test_capture(lib):
    n = Note(lib)
    n.produce()
    assert n.product(A, capture=4)       # an eager producer runs before or after the whole graph ...
    assert not n.product(A)              # ... and what was recorded is no answer for the stream
    n.produce(capture=5)
    assert n.product(A) and n.product(B, capture=6)   # nor is a recorded producer a matter of other captures or of eager calls
    assert not n.product(B, capture=5)                # a second stream of the capture
    assert not n.product(A, capture=5) and n.product(A, capture=5)
    n.produce(capture=5)
    assert not n.product(A, capture=5) and n.product(A, capture=5)
    # more captures with producers than are held: one that is no longer known is held back, once, as is every new one
    for c in range(100, 140):
        n.produce(capture=c)
    assert not n.product(A, capture=5) and not n.product(A, capture=139) and n.product(A, capture=139)
    assert not n.product(A, capture=200) and n.product(A, capture=200)
    assert n.product(A)


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
    # a producer whose stream cannot say concerns everything
    n.produce(capture=5)
    assert not n.product(A, capture=5) and n.product(A, capture=5) and n.product(A, capture=6)
    n.produce(known=False)
    assert not n.product(A) and not n.product(A, capture=5) and not n.product(A, capture=6)


def test_two_threads_on_one_stream(lib):
    # a product between a producer's two marks, and one that begins before another's launch
    n = Note(lib)
    n.mark()
    assert not n.product(A)
    n.mark()
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
    # early <=> a product of the same key was launched without the early start, after it had begun behind the last mark of every producer
    # of the same capture (or, for eager products, of every eager one).  (With more keys than are held, entries are forgotten: then only =>.)
    rng = random.Random(seed)
    n = Note(lib)
    captures = (0, 0, 7, 8) if keys < 100 else range(60)
    names = [(rng.randrange(2), 0x100 * (i + 1), rng.choice(captures)) for i in range(keys)]
    open_products, settled, last_mark, early_count = [], {}, {}, 0

    def end(i, launched):
        p, key, t, early = open_products.pop(i)
        lib.product_end(p, launched)
        if launched and not early and t > last_mark.get(key[2], 0):
            settled[key] = t

    for now in range(1, 6000 if keys < 100 else 20000):
        what = rng.random()
        if what < (0.15 if keys < 100 else 0.005):
            c = rng.choice(captures)
            n.mark(capture=c)
            last_mark[c] = now
        elif what < 0.4 and open_products:
            end(rng.randrange(len(open_products)), rng.random() < 0.9)
        else:
            key = rng.choice(names)
            p, early = n.begin(key[1], device=key[0], capture=key[2])
            allowed = last_mark.get(key[2], 0) == 0 or settled.get(key, 0) > last_mark[key[2]]
            assert (early == allowed) if keys < 100 else (allowed or not early)
            early_count += early
            open_products.append((p, key, now, early))
            if len(open_products) > 4:
                end(0, True)
    assert early_count > 100
    while open_products:
        end(0, False)


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
        assert api.count(launch) == 1 and re.search(r"const bd::Producing producing\(g_producers, [^\n]*stream_key\(d\.device, [^\n]*\n\s+if \(" + re.escape(launch), api)
    assert len(re.findall(r"bd::ProductStart start\(", api)) == api.count("start.launched();") == 2
