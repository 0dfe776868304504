"""First touch of result pages: every page is there afterwards, nothing outside
the array changes, and memory that cannot be written is left to the copy."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1601_03815_gb300", "csrc")

PROGRAM = r"""
#include "host_pages.h"
int main() {
    const size_t n = (size_t(50) << 20) + 12345, page = sysconf(_SC_PAGESIZE);
    char* p = (char*)mmap(0, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    p[2] = p[n - 1] = 5;
    {
        kin::HostPages h(p + 3, n - 4);
        h.wait(n - 4);
    }
    std::vector<unsigned char> in((n + page - 1) / page);
    mincore(p, n, in.data());
    for (unsigned char c : in)
        if (!(c & 1)) return 1;
    if (p[2] != 5 || p[n - 1] != 5) return 2;
    char* r = (char*)mmap(0, n, PROT_READ, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    kin::HostPages h(r, n);
    h.wait(n);
    return 0;
}
"""


def test_pages_are_touched(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0
