"""Which page-locked result arrays fdllm_select_host lets the GPU write in place: those mapped as a
whole.  The decision (csrc/host_view.h) runs on the host against a table of locked pages."""
import os
import shutil
import subprocess

import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PAGE = 4096

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "host_view.h"

// argv: page map (one character per page: '.' not locked, a letter a mapping of its own), then
// pairs of offset and bytes; prints 1 where the array is one mapping, 0 otherwise.
int main(int argc, char **argv)
{
    const char *map = argv[1];
    const int64_t page = %d, pages = (int64_t)strlen(map);
    uint8_t *const base = (uint8_t *)(uintptr_t)0x10000000;
    auto device_of = [&](uint8_t *p) -> uint8_t * {
        const int64_t at = p - base;
        if (at < 0 || at >= pages * page)
            exit(9);  // looked outside the array's pages
        const char c = map[at / page];
        return c == '.' ? nullptr : p + (uintptr_t)(c - 'a' + 1) * 0x1000000000;
    };
    for (int i = 2; i + 1 < argc; i += 2) {
        uint8_t *const host = base + atoll(argv[i]);
        uint8_t *const d = fdllm::whole_view(host, atoll(argv[i + 1]), page, device_of);
        if (d && d != device_of(host))
            return 8;
        printf("%%d", d != nullptr);
    }
    return 0;
}
""" % PAGE


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("host_view")
    (d / "main.cpp").write_text(PROGRAM)
    include = os.path.join(ROOT, "paper_2606_02955_gb300", "csrc")
    subprocess.run([cxx, "-std=c++17", "-I", include, str(d / "main.cpp"), "-o", str(d / "main")],
                   check=True)
    return str(d / "main")


@pytest.mark.parametrize("pages", ["a", "aa", "ab", "a.a", "aba", "aaa", "aa.aa", ".aa", "aaaaa"])
def test_in_place_only_where_every_page_is_mapped(program, pages):
    end = len(pages) * PAGE
    arrays = [(o, n) for o in (0, 1, 4, PAGE - 1, PAGE, PAGE + 1, 2 * PAGE - 4)
              for n in (1, 4, PAGE - 1, PAGE, PAGE + 1, 2 * PAGE, 2 * PAGE + 4, end - o)
              if o + n <= end and n > 0]
    out = subprocess.run([program, pages] + [str(v) for a in arrays for v in a],
                         check=True, capture_output=True, text=True).stdout
    for (o, n), got in zip(arrays, out):
        touched = pages[o // PAGE:(o + n - 1) // PAGE + 1]
        assert got == str(int(len(set(touched)) == 1 and touched[0] != ".")), (pages, o, n)


@pytest.mark.gpu
def test_results_in_an_array_locked_at_both_ends(fd):
    """Tokens in memory whose first and last 64 KB are page-locked and whose middle is not are not
    written in place; the runtime then refuses the copy that spans them, and nothing is written."""
    import ctypes
    import mmap
    import numpy as np
    B, L, V = 64, 1024, 64
    end = 65536
    buf = np.frombuffer(mmap.mmap(-1, B * L * 4), np.uint8)
    rt = torch.cuda.cudart()
    ends = [buf.ctypes.data, buf.ctypes.data + buf.size - end]
    assert all(int(rt.cudaHostRegister(p, end, 0)) == 0 for p in ends)
    try:
        x = torch.randn(B, L, V, generator=torch.Generator().manual_seed(6)).to(torch.bfloat16)
        mask = torch.ones(B, L, dtype=torch.uint8)
        tok = torch.from_numpy(buf.view(np.int32)).view(B, L)
        tok.fill_(-1)
        commit = torch.zeros(B, L, dtype=torch.uint8).pin_memory()
        n = torch.zeros(B, dtype=torch.int32).pin_memory()
        px = x.pin_memory()
        with pytest.raises(fd.FdllmError) as e:
            fd.fdllm_select(px, mask, 0.5, "threshold", tok, commit, n)
        assert e.value.status == fd.ERR_CUDA
        ctypes.CDLL(fd.library_path()).cudaGetLastError()  # the refused copy, for the calls below
        torch.cuda.synchronize()
        assert (tok == -1).all() and (commit == 0).all() and (n == 0).all() and (mask == 1).all()
        tok = torch.full((B, L), -1, dtype=torch.int32).pin_memory()
        fd.fdllm_select(px, mask, 0.5, "threshold", tok, commit, n)
        assert (n > 0).all() and torch.equal(tok >= 0, commit != 0)
    finally:
        for p in ends:
            rt.cudaHostUnregister(p)
