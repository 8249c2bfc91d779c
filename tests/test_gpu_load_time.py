"""GPU: what the bank order of a general code of check degree 6 adds to load_code().
The same code less one edge has no such order; made in line, the order took two thirds
of the call on top."""
import time

import numpy as np
import pytest

import paper_2208_05795_gb300 as tsx
import synth

pytestmark = pytest.mark.gpu


def test_load_time_of_a_degree_six_code():
    n, m = 4000, 2000
    rng = np.random.default_rng(1)
    cols = np.concatenate([np.sort(rng.choice(n, 6, replace=False)) for _ in range(m)]).astype(np.int32)
    ptr = np.arange(0, 6 * m + 1, 6, dtype=np.int32)
    less = ptr.copy()
    less[-1] -= 1
    codes = [synth.csr_code(n, m, ptr, cols), synth.csr_code(n, m, less, cols[:-1])]
    best = [1e9, 1e9]
    for _ in range(12):
        for i, c in enumerate(codes):
            t = time.perf_counter()
            tsx.load_code(c)
            best[i] = min(best[i], time.perf_counter() - t)
    assert best[0] < 1.35 * best[1], best
