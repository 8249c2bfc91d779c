"""The bank order of a general code's checks (csrc/banks.h, host code): every
row is there once with its own variable nodes, and where banks are met at
random over many warps an access takes at most 2 wavefronts on average (3.4
in the matrix's order).  The header is compiled with g++ as it stands."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r'''
#include <cstdio>
#include "banks.h"
int main() {
    int m, dc;
    if (scanf("%d %d", &m, &dc) != 2) return 1;
    std::vector<uint16_t> col(m * dc);
    for (auto &x : col) { unsigned v; if (scanf("%u", &v) != 1) return 1; x = (uint16_t)v; }
    for (uint16_t x : tsx::bank_order(m, dc, col)) printf("%u\n", x);
}
'''


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("banks")
    (d / "main.cpp").write_text(MAIN)
    exe = str(d / "main")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2208_05795_gb300", "csrc"),
                    str(d / "main.cpp"), "-o", exe], check=True)
    return exe


def _wavefronts(rows):
    """Mean over (warp of 32 rows, position) of the most words any bank is asked for."""
    w = []
    for g in range(0, len(rows), 32):
        for p in range(rows.shape[1]):
            v = np.unique(rows[g:g + 32, p])
            w.append(np.bincount(v % 32).max())
    return np.mean(w)


@pytest.mark.parametrize("n,m,dc", [(12, 1, 6), (40, 31, 6), (40, 32, 6), (64, 33, 6), (200, 100, 6), (1008, 504, 6),
                                    (4000, 2000, 6), (32, 96, 6), (300, 64, 4)])
@pytest.mark.parametrize("kind", ["random", "one_bank"])
def test_bank_order(program, n, m, dc, kind):
    rng = np.random.default_rng(n + m)
    pool = np.arange(n) * (32 if kind == "one_bank" else 1)  # one_bank: nothing to gain, every edge in bank 0
    rows = np.stack([np.sort(rng.choice(pool, dc, replace=False)) for _ in range(m)])
    if rows.max() > 65535:
        rows %= 65536
    text = "%d %d\n%s\n" % (m, dc, "\n".join(map(str, rows.ravel())))
    out = subprocess.run([program], input=text, capture_output=True, text=True, check=True, timeout=60).stdout
    got = np.array(out.split(), dtype=np.int64).reshape(m, dc)
    assert sorted(map(tuple, np.sort(got, axis=1))) == sorted(map(tuple, np.sort(rows, axis=1)))
    if kind == "random" and m >= 500:
        assert _wavefronts(got) <= 2.0 < _wavefronts(rows)
