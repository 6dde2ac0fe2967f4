"""Output pages are made present before a copy from the device; an address where nothing
is mapped (a device pointer handed to a read-out) is left for the copy to refuse."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1906_04722_gb300", "csrc")
PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include "lbm_host.h"
int main(int argc, char** argv) {
    const size_t n = (size_t(7) << 20) + 123;
    if (std::strcmp(argv[1], "unmapped") == 0) {
        lbmk::touch_pages((char*)0x200000000, n);
        return 0;
    }
    char* p = (char*)mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    if (std::strcmp(argv[1], "present") == 0) std::memset(p, 7, n);
    lbmk::touch_pages(p, n);
    unsigned char there[1 << 16];
    if (mincore(p, n, there) != 0) return 1;
    const size_t page = (size_t)sysconf(_SC_PAGESIZE);
    for (size_t i = 0; i < (n + page - 1) / page; ++i)
        if (!(there[i] & 1)) return 2;
    for (size_t i = 0; i < n; ++i)
        if (p[i] != (argv[1][0] == 'p' ? 7 : 0)) return 3;
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("pages")
    src, exe = str(d / "pages.cpp"), str(d / "pages")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", CSRC, src, "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("pages", ["fresh", "present", "unmapped"])
def test_touch_pages(program, pages):
    assert subprocess.run([program, pages]).returncode == 0
