"""Room in a list that many warps fill (reserve.cuh), compiled for the host:
requests whose sum passes 2^32 are granted while they fit, never point outside
the list, and leave every entry below its length either stored or marked empty,
once.  CPU only."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#define CT_HD inline
#include "reserve.cuh"
#include <cstdio>
#include <vector>
int main() {
    for (int cap : {1, 1000, 1 << 20}) {
        std::vector<unsigned char> written(cap, 0);
        unsigned long long count = 0;
        unsigned r = 12345u;
        for (int i = 0; i < 600000; ++i) {
            r = r * 1664525u + 1013904223u;
            const int n = i % 3 == 0 ? 16384 : (int)(r >> (i % 5 == 1 ? 30 : 18));
            const ct::ListRoom room = ct::list_room(count, n, cap);
            if (room.fits != (count + n <= (unsigned long long)cap)) return 1;
            count += n;
            if (room.begin < 0 || room.begin > cap) return 2;
            const int end = room.fits ? room.begin + n : cap;
            if (end > cap) return 3;
            for (int k = room.begin; k < end; ++k)
                if (written[k]++) return 4;
        }
        if (count < (1ull << 32)) return 5;
        if (ct::list_length(count, cap) != cap || ct::list_length(cap - 1, cap) != cap - 1) return 6;
        for (int k = 0; k < cap; ++k)
            if (!written[k]) return 7;
    }
    puts("ok");
    return 0;
}
"""


def test_counts_past_32_bits(tmp_path):
    src, exe = tmp_path / "reserve.cpp", tmp_path / "reserve"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2510_14147_gb300", "csrc"),
                    "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], stdout=subprocess.PIPE)
    assert out.returncode == 0 and out.stdout == b"ok\n"
