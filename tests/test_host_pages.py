"""Host pages that a device copy is about to write: made present once, their contents kept, and
left alone when they are there already."""
import ctypes
import mmap
import os
import subprocess

import numpy as np
import pytest

from conftest import ROOT

PAGE = mmap.PAGESIZE


@pytest.fixture(scope="module")
def populate(tmp_path_factory):
    d = tmp_path_factory.mktemp("pages")
    src, lib = d / "pages.cpp", d / "libpages.so"
    src.write_text('#include "host_pages.h"\n'
                   'extern "C" size_t populate(void* p, size_t n) { return lbm::populate_host_pages(p, n); }\n')
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread", "-I",
                    os.path.join(ROOT, "paper_2608_13437_gb300", "csrc"), str(src), "-o", str(lib)], check=True)
    f = ctypes.CDLL(str(lib)).populate
    f.restype, f.argtypes = ctypes.c_size_t, [ctypes.c_void_p, ctypes.c_size_t]
    return f


def _fresh(pages):
    m = mmap.mmap(-1, pages * PAGE)
    a = np.frombuffer(m, dtype=np.uint8)
    return m, a, a.ctypes.data


# one thread and several, one look at the pages and several
@pytest.mark.parametrize("pages", [5, 700, 2048, 5000])
def test_pages_are_asked_for_once(populate, pages):
    m, a, at = _fresh(pages)
    assert populate(at, pages * PAGE) == pages
    assert populate(at, pages * PAGE) == 0
    a[:] = 7
    assert populate(at + 1, pages * PAGE - 1) == 0 and (a == 7).all()


@pytest.mark.parametrize("pages,touched", [(64, 10), (5000, 2047), (5000, 2048), (5000, 4096)])
def test_pages_from_the_first_missing_one(populate, pages, touched):
    m, a, at = _fresh(pages)
    a[:touched * PAGE] = 3
    assert populate(at, pages * PAGE) == pages - touched
    assert (a[:touched * PAGE] == 3).all() and (a[touched * PAGE:] == 0).all()
    assert populate(at, pages * PAGE) == 0


def test_ends_within_a_page_and_short_ranges_are_left_alone(populate):
    m, a, at = _fresh(16)
    assert populate(at, 3 * PAGE) == 0
    assert populate(at + 1, 5 * PAGE) == 4  # the whole pages inside
