"""Rows of a list to the host (csrc/rows.h, host code): one 2-D copy up to a
pitch that every device takes, single copies of the rows beyond.  The header is
compiled with g++ as it stands, with copies that note what they were asked for."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r'''
#include <cstdio>
#include "rows.h"
int main() {
    unsigned long long pitch, width, rows, bad;
    while (scanf("%llu %llu %llu %llu", &pitch, &width, &rows, &bad) == 4) {
        char *dst = (char *)4096, *src = (char *)8192;
        unsigned long long calls = 0;
        const int e = tsx::copy_rows(dst, src, pitch, width, rows,
            [&](void *d, size_t dp, const void *s, size_t sp, size_t w, size_t n) {
                printf("2d %td %zu %td %zu %zu %zu;", (char *)d - dst, dp, (const char *)s - src, sp, w, n);
                return 0;
            },
            [&](void *d, const void *s, size_t n) {
                printf("1d %td %td %zu;", (char *)d - dst, (const char *)s - src, n);
                return ++calls == bad ? 7 : 0;
            });
        printf("%d\n", e);
    }
}
'''


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    (d / "main.cpp").write_text(MAIN)
    exe = str(d / "main")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2208_05795_gb300", "csrc"),
                    str(d / "main.cpp"), "-o", exe], check=True)
    return lambda *a: subprocess.run([exe], input="%d %d %d %d\n" % a, capture_output=True, text=True, check=True).stdout.strip()


@pytest.mark.parametrize("pitch", [256, 4 * 11_700_000, 2 ** 30])
def test_one_copy(program, pitch):
    assert program(pitch, 40, 6, 0) == "2d 0 40 0 %d 40 6;0" % pitch


@pytest.mark.parametrize("pitch", [2 ** 30 + 256, 2 ** 31, 2 ** 33])
def test_beyond_the_pitch_limit_row_by_row(program, pitch):
    assert program(pitch, 40, 3, 0) == "".join("1d %d %d 40;" % (40 * r, pitch * r) for r in range(3)) + "0"
    assert program(pitch, 40, 3, 2).endswith(";7") and program(pitch, 40, 3, 2).count("1d") == 2


def test_the_library_copies_rows_this_way():
    text = open(os.path.join(ROOT, "paper_2208_05795_gb300", "csrc", "api.cu")).read()
    assert text.count("cudaMemcpy2D(") == 1 and text.count("fetch_rows(") == 3
