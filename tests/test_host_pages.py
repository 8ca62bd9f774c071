"""Mapping the pages of a host output buffer ahead of the GPU's copy
(csrc/host_pages.h) changes nothing a program can see: it does not store into
the buffer, whose bytes may still be the source of a copy queued earlier on the
stream, and an address that cannot be written stays an error of the copy.

The buffer here reaches from writable pages into a read-only one, so the
kernel's advice is refused; the call runs in a child process, which a store into
the read-only page would end.
"""
import multiprocessing as mp
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """
#include "host_pages.h"
extern "C" int run(int writable, int locked) {
    const size_t page = (size_t)sysconf(_SC_PAGESIZE), n = (size_t)(writable + locked) * page;
    char* p = static_cast<char*>(mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0));
    if (p == MAP_FAILED) return -1;
    for (size_t k = 0; k < n; ++k) p[k] = 7;
    if (locked && mprotect(p + writable * page, (size_t)locked * page, PROT_READ)) return -1;
    eulbfs::map_output(p + 16, n - 16);
    int changed = 0;
    for (size_t k = 0; k < n; ++k) changed += p[k] != 7;
    return changed;
}
"""


def _call(path, writable, locked, q):
    import ctypes
    q.put(ctypes.CDLL(path).run(writable, locked))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("pages")
    src, out = d / "pages.cpp", d / "pages.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2507_03366_gb300", "csrc"), str(src), "-o", str(out)], check=True)
    return str(out)


@pytest.mark.parametrize("writable,locked", [(64, 0), (64, 1), (1, 64)])
def test_buffer_keeps_its_bytes(lib, writable, locked):
    ctx = mp.get_context("spawn")
    q = ctx.Queue()
    p = ctx.Process(target=_call, args=(lib, writable, locked, q))
    p.start()
    p.join(60)
    assert p.exitcode == 0
    assert q.get(timeout=10) == 0
