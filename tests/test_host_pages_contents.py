"""Pages made present ahead of a read-out keep what they hold, and a page in the
middle of the result that may not be written is left to the copy (whose error the
read-out then returns) together with nothing but its own range."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1601_03815_gb300", "csrc")

PROGRAM = r"""
#include "host_pages.h"
#include <cstdio>
int main() {
    const size_t n = size_t(50) << 20, page = sysconf(_SC_PAGESIZE), at = size_t(20) << 20;
    // a read-only page, then a hole, in the middle of a part
    for (int hole = 0; hole < 2; ++hole) {
        char* p = (char*)mmap(0, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
        if (p == MAP_FAILED) return 10;
        if (hole ? munmap(p + at, page) : mprotect(p + at, page, PROT_READ)) return 11;
        {
            kin::HostPages h(p, n);
            h.wait(n);
        }
        munmap(p, n);
    }
    // a file of ones: present or not, its bytes are those of the file afterwards
    FILE* f = tmpfile();
    std::vector<char> ones(1 << 20, 1);
    for (size_t k = 0; k < n; k += ones.size())
        if (fwrite(ones.data(), 1, ones.size(), f) != ones.size()) return 12;
    fflush(f);
    char* q = (char*)mmap(0, n, PROT_READ | PROT_WRITE, MAP_PRIVATE, fileno(f), 0);
    if (q == MAP_FAILED) return 13;
    posix_fadvise(fileno(f), 0, 0, POSIX_FADV_DONTNEED);
    // and memory whose present pages are not those that are looked at
    char* a = (char*)mmap(0, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    for (size_t k = page; k < n; k += 2 * page) a[k] = a[k + 7] = 1;
    madvise(a, page, MADV_DONTNEED);
    {
        kin::HostPages h(q, n), g(a, n);
        h.wait(n);
        g.wait(n);
    }
    // what is there needs no parts: the copy is one
    if (kin::HostPages(a, n).pending()) return 4;
    for (size_t k = 0; k < n; k += 64)
        if (q[k] != 1) return 2;
    for (size_t k = page; k < n; k += 2 * page)
        if (a[k] != 1 || a[k + 7] != 1) return 3;
    return 0;
}
"""


def test_pages_keep_their_contents_and_protected_pages_are_left(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text("#include <fcntl.h>\n" + PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0
