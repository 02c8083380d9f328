"""The word loads of the sin^2 convolution (row_words.cuh), run on the host with
counting loads: no byte outside the label array is read, every word is
aligned, and the words hold the row's cells."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include "row_words.cuh"
int main()
{
    alignas(64) static unsigned char buf[4096];
    long checked = 0;
    for (int nz = 1; nz <= 40; ++nz)
        for (int off = 0; off < 8; ++off)
            for (int rows = 1; rows <= 5; ++rows) {
                unsigned char *a = buf + 64 + off, *e = a + rows * nz;
                memset(buf, 0xff, sizeof buf);
                for (int k = 0; k < rows * nz; ++k) a[k] = (unsigned char)(1 + k % 250);
                bool bad = false;
                auto word = [&](uintptr_t p) {
                    bad |= p % 8 != 0 || p < (uintptr_t)a || p + 8 > (uintptr_t)e;
                    uint64_t w;
                    memcpy(&w, (void *)p, 8);
                    return w;
                };
                auto byte = [&](uintptr_t p) {
                    bad |= p < (uintptr_t)a || p >= (uintptr_t)e;
                    return *(unsigned char *)p;
                };
                for (int r = 0; r < rows; ++r)
                    for (int k0 = 0; k0 < nz; k0 += 8) {
                        uint64_t w[3];
                        vesis::row_words((uintptr_t)a, (unsigned)(r * nz), k0, nz, (unsigned)(e - a),
                                         word, byte, w[0], w[1], w[2]);
                        for (int c = -8; c < 16; ++c) {
                            const int k = k0 + c;
                            const unsigned want = k >= 0 && k < nz ? a[r * nz + k] : 0u;
                            const unsigned got = (unsigned)(w[(c + 8) / 8] >> (8 * ((c + 8) % 8))) & 0xffu;
                            if (want != got || bad) {
                                printf("nz %d off %d rows %d row %d cell %d: %u, not %u%s\n", nz, off, rows,
                                       r, k, got, want, bad ? " (read outside)" : "");
                                return 1;
                            }
                            ++checked;
                        }
                    }
            }
    printf("%ld\n", checked);
    return 0;
}
"""


def test_row_words_read_the_array_alone(tmp_path):
    src, exe = tmp_path / "words.cpp", tmp_path / "words"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Wno-unknown-pragmas", "-Werror", "-I",
                    os.path.join(ROOT, "paper_2208_05524_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 100000
