"""CPU check of the loads of packed rows that are no 16-byte multiples (csrc/ragged_piece.h, the code the
unpack and repack kernels run): built for the host with the address sanitizer and run over samples that
end exactly where their allocation ends, so a read past them is an error even inside an aligned word."""
import pathlib
import subprocess

import pytest

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_0906_1887_gb300" / "csrc"

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "ragged_piece.h"
int main() {
    for (int row_bytes = 1; row_bytes <= 150; row_bytes += row_bytes < 36 ? 1 : 19)
        for (int rows = 1; rows <= 9; ++rows) {
            const int n = rows * row_bytes;
            unsigned char* p = static_cast<unsigned char*>(malloc(n));   // 16-byte aligned; ends at the last sample
            for (int k = 0; k < n; ++k) p[k] = (unsigned char)(37 * k + 11);
            for (int r = 0; r < rows; ++r)
                for (int c = 0; c * 16 < row_bytes; ++c)
                    for (int whole = 0; whole < 2; ++whole) {
                        const int off = r * row_bytes + 16 * c, left = row_bytes - 16 * c < 16 ? row_bytes - 16 * c : 16;
                        uint32_t v[4];
                        corr::load_piece(p, off, n, whole ? 16 : left, corr::tail_word(p, n), v);   // as the repack / the unpack asks for it
                        for (int b = 0; b < 16; ++b) {
                            const unsigned got = (v[b >> 2] >> (8 * (b & 3))) & 255u;
                            if (b < left ? got != p[off + b] : (!whole && got)) return 1;
                        }
                    }
            free(p);
        }
    puts("ok");
}
"""


def test_ragged_loads_stay_inside_the_samples(tmp_path):
    src, exe = tmp_path / "m.cpp", tmp_path / "m"
    src.write_text(MAIN)
    cmd = ["g++", "-std=c++17", "-O1", "-g", "-fsanitize=address", "-I", str(CSRC), str(src), "-o", str(exe)]
    b = subprocess.run(cmd, capture_output=True, text=True)
    if b.returncode != 0 and "asan" in b.stderr:
        pytest.skip("no address sanitizer runtime")
    assert b.returncode == 0, b.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stderr[:2000]
