"""Room in a list that many warps fill (reserve.cuh), compiled for the host:
requests whose sum passes 2^31 and other warps that take room in between never
bring the count past the list's end, and every request that fits is granted.
CPU only."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#define CT_HD inline
#include "reserve.cuh"
#include <cstdio>
int main() {
    const int cap = 1 << 20;
    int count = 0;
    unsigned long long asked = 0;
    unsigned r = 12345u;
    for (int i = 0; i < 300000; ++i) {
        r = r * 1664525u + 1013904223u;
        const int n = i % 3 == 0 ? 16384 : (int)(r >> 18);   // 0 .. 16383
        const int seen = i % 5 ? count : 0;                  // a count read long ago
        int others = (int)((r >> 8) & 3u);                   // other warps take an entry each first
        const int before = count;
        int taken = 0;
        const int at = ct::list_reserve(seen, n, cap, [&](int expected, int desired) {
            if (others > 0 && count < cap) { --others; ++count; ++taken; }
            const int found = count;
            if (found == expected) count = desired;
            return found;
        });
        asked += (unsigned)n;
        if (at >= 0 && (at != before + taken || count != at + n)) return 1;
        if (at < 0 && n <= cap - count) return 2;
        if (count < 0 || count > cap) return 3;
    }
    if (asked < (1ull << 31)) return 4;
    printf("%d\n", count);
    return 0;
}
"""


def test_count_never_passes_the_end(tmp_path):
    src, exe = tmp_path / "reserve.cpp", tmp_path / "reserve"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2510_14147_gb300", "csrc"),
                    "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], stdout=subprocess.PIPE)
    assert out.returncode == 0
    assert 0 < int(out.stdout) <= 1 << 20
