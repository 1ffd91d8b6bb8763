"""Touching a destination's pages leaves every byte as it was, from any start
and for any length (host only)."""

import os
import subprocess
import tempfile

SRC = r"""
#include "host_pages.h"
#include <cstdio>
#include <cstring>
int main() {
    const size_t cap = 9u << 20;
    for (size_t off : {0ul, 1ul, 4095ul, 65537ul})
        for (size_t len : {0ul, 1ul, (2ul << 20) - 1, 2ul << 20, (5ul << 20) + 4097}) {
            for (int fresh = 0; fresh < 2; ++fresh) {
                unsigned char *p = (unsigned char *)mmap(nullptr, cap, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
                if (!fresh) for (size_t i = 0; i < cap / 2; ++i) p[i] = (unsigned char)(i * 37 + 11);   // half backed
                hydro::touch_pages(p + off, len);
                for (size_t i = 0; i < cap; ++i)
                    if (p[i] != (fresh || i >= cap / 2 ? 0 : (unsigned char)(i * 37 + 11))) return printf("%zu %zu %zu\n", off, len, i), 1;
                munmap(p, cap);
            }
        }
    hydro::touch_pages(nullptr, 1u << 30);
    // a read-only and a vanished mapping: nothing happens
    unsigned char *p = (unsigned char *)mmap(nullptr, cap, PROT_READ, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    hydro::touch_pages(p, cap);
    munmap(p, cap);
    hydro::touch_pages(p, cap);
    return 0;
}
"""


def test_touch_pages_keeps_contents():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "t.cpp"), os.path.join(d, "t")
        with open(src, "w") as f:
            f.write(SRC)
        subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", os.path.join(root, "paper_1510_05061_gb300", "csrc"),
                        src, "-o", exe], check=True)
        r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, r.stdout
