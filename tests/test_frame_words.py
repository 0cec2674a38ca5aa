"""The frame words the word path of the 1-bit ingest copies (csrc/frame_words.cuh,
compiled here for the host): every pixel of the region is covered, and the whole words
and the bytes behind them end with the region's last byte, where the caller's buffer
may end."""

import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2407_20692_gb300", "csrc")

PROGRAM = r"""
#include "frame_words.cuh"
#include <cstdio>
#include <cstdlib>
struct Frames { int height, width, x0, y0; int64_t row_stride; };
int main() {
    std::srand(5);
    for (int t = 0; t < 20000; ++t) {
        Frames d;
        d.height = 1 + std::rand() % 9, d.width = 1 + std::rand() % (t % 2 ? 40 : 200);
        d.x0 = std::rand() % 70, d.y0 = std::rand() % 4;
        d.row_stride = d.x0 + d.width + (t % 3 ? std::rand() % 8 : std::rand() % 5000);
        const int64_t last = (int64_t)(d.y0 + d.height - 1) * d.row_stride + d.x0 + d.width - 1;
        const int64_t w0 = cpi::region_first_word(d), w1 = cpi::region_last_word(d);
        const int64_t whole = cpi::region_whole_words(d);
        const int rest = cpi::region_rest_bytes(d);
        if (rest < 0 || rest > 3 || 4 * whole + rest != last / 8 + 1) return std::printf("not up to the last pixel\n"), 1;
        if (rest ? whole != w1 : whole != w1 + 1) return std::printf("the partial word is not the last\n"), 1;
        for (int y = 0; y < d.height; ++y)
            for (int x = 0; x < d.width; ++x) {
                const int64_t w = ((d.y0 + y) * d.row_stride + d.x0 + x) >> 5;
                if (w < w0 || w > w1) return std::printf("pixel not covered\n"), 1;
            }
    }
    // rows far apart: the words between them would be read for nothing
    const Frames narrow{64, 8, 0, 0, 128}, apart{64, 8, 0, 0, 512}, wide{64, 31, 0, 0, 512}, lone{16, 50, 0, 0, 8192};
    if (!cpi::words_pay(narrow, narrow) || cpi::words_pay(apart, apart) || !cpi::words_pay(wide, wide) ||
        cpi::words_pay(lone, lone) || !cpi::words_pay(wide, apart))
        return std::printf("words_pay\n"), 1;
    return 0;
}
"""


def test_words_cover_the_region_end_with_it_and_pay(tmp_path):
    src, exe = tmp_path / "words.cpp", tmp_path / "words"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    done = subprocess.run([str(exe)], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout


def test_the_kernel_copies_by_that_count():
    body = open(os.path.join(CSRC, "ingest.cu")).read()
    body = body[body.index("ingest_bits_kernel("):]
    body = body[:body.index("cp.async.wait_all")]
    assert "region_whole_words(d)" in body and "frame_stride >> 2" not in body
